"""The fp32 layer kernel through the C ABI against the CPU oracle, at the sizes where its tiling changes.  Needs a B200."""
import ctypes

import numpy as np
import pytest
import torch

import dsvt_inputs as di
from gpu_helpers import check_close, dev, rowoff_of, upload_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,grid,window,tau,C,heads,hidden,option", [
    (1, 24, 12, 36, 128, 8, 0, ""),           # one voxel: one row, blocks without work
    (9, 12, 12, 36, 192, 8, 192, "pe"),       # one set of nine rows: 8-row groups of a thread tile
    (144, 12, 12, 36, 192, 8, 384, ""),       # one full window: four sets of 36 rows, one per tile
    (560, 24, 12, 64, 192, 8, 384, "rpb"),    # fewer rows than blocks x set size; sets of up to 64 rows, a tile's most
    (3000, 60, 30, 96, 128, 4, 256, ""),      # tiles of up to 96 rows, head dim 32
    (9000, 100, 12, 36, 64, 4, 128, "pe"),    # several tiles per block
    (20000, 150, 12, 36, 128, 8, 128, "rpb"),
    (700, 36, 12, 36, 192, 8, 256, ""),       # a deep second product of four chunks
    (14001, 150, 12, 36, 192, 8, 64, "pe"),   # two passes; the narrowest tile of the first MLP product
    (45000, 240, 12, 48, 64, 4, 64, ""),      # two passes of many tiles per block
])
def test_layer_fp32_matches_oracle(oracle, n, grid, window, tau, C, heads, hidden, option):
    from paper_2301_06051_b200 import api

    case = di.random_case(n + C, n, (grid, grid, 1), (window, window, 1), tau, C, heads, hidden, layernorm=hidden > 0)
    layer = case["blocks"][0][0]
    rng = np.random.default_rng(n)
    pe = rng.standard_normal((n, C)).astype(np.float32) if option == "pe" else None
    if option == "rpb":
        layer["rpb"] = rng.standard_normal((heads, (2 * window - 1) ** 2)).astype(np.float32)
        layer["rpb_extent"] = (window, window, 1)
    ctx = api.Context(n, (-(-grid // window)) ** 2, C)
    coords, x = dev(case["coords"]), dev(case["feats"])
    table = ctx.partition(coords, 1, case["grid"], case["window"], tau, 0)
    w = api.device_weights(layer, api.FP32, ctx.device)
    y = torch.empty_like(x)
    ctx.layer(x, table, w, y, pe=None if pe is None else dev(pe), coords=coords)
    assert ctx.status_sync() == 0
    p = oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0)
    want = oracle.layer(case["feats"], p.set_table, layer, pe=pe, coords=case["coords"])
    check_close(y.cpu().numpy(), want, "fp32", "n=%d C=%d" % (n, C))
    z = x.clone()  # in place: a tile's rows are its own
    ctx.layer(z, table, w, z, pe=None if pe is None else dev(pe), coords=coords)
    assert ctx.status_sync() == 0 and torch.equal(y, z)


@pytest.mark.parametrize("C,heads,hidden", [(128, 8, 0), (192, 8, 384)])
def test_row_offsets_that_claim_more_rows_than_a_set_has(oracle, C, heads, hidden):
    """Caller-made row offsets with room for seven members that their set does not have: DSVT_STATUS_BAD_INDEX, and the
    voxels of all other sets come out right."""
    from paper_2301_06051_b200 import api

    n, tau = 700, 36
    case = di.random_case(C, n, (48, 48, 1), (12, 12, 1), tau, C, heads, hidden, layernorm=hidden > 0)
    layer = case["blocks"][0][0]
    p = oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0)
    table = upload_table(p.set_table)
    long = len(p.set_table) // 2
    table.set_rowoff[long + 1 : len(p.set_table) + 1] += 7
    ctx = api.Context(n, 16, C)
    x = dev(case["feats"])
    y = torch.empty_like(x)
    ctx.layer(x, table, api.device_weights(layer, api.FP32, ctx.device), y)
    assert ctx.status_sync() == api.STATUS_BAD_INDEX
    others = np.setdiff1d(np.arange(n), p.set_table[long])
    want = oracle.layer(case["feats"], p.set_table, layer)
    check_close(y.cpu().numpy()[others], want[others], "fp32", "the other sets")


@pytest.mark.parametrize("tau,C,heads,hidden", [(36, 192, 8, 384), (36, 192, 8, 256), (36, 192, 8, 0), (36, 128, 8, 256), (90, 128, 4, 0),
                                                (36, 64, 4, 128)])
def test_layer_fp32_is_as_precise_as_fp32(oracle, tau, C, heads, hidden):
    """One layer against float64.  Sums of 64 to 384 products with a rounding of 2^-24 each, two to four of them in a chain, come
    to 1e-7 ... 3e-7 of the result (2-norm); the bounds are 4e-7 and 12 times that for the largest error, where operands of
    two bfloat16 parts (2^-17) show 5e-6."""
    from paper_2301_06051_b200 import api

    n = 1500
    case = di.random_case(C + hidden, n, (72, 72, 1), (12, 12, 1), tau, C, heads, hidden, layernorm=hidden > 0)
    layer = case["blocks"][0][0]
    ctx = api.Context(n, 36, C)
    x = dev(case["feats"])
    table = ctx.partition(dev(case["coords"]), 1, case["grid"], case["window"], tau, 0)
    y = torch.empty_like(x)
    ctx.layer(x, table, api.device_weights(layer, api.FP32, ctx.device), y)
    assert ctx.status_sync() == 0
    want = oracle.layer(case["feats"], oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0).set_table, layer)
    err = y.cpu().numpy().astype(np.float64) - want
    assert np.linalg.norm(err) <= 4e-7 * np.linalg.norm(want)
    assert np.abs(err).max() <= 5e-6 * np.sqrt((want ** 2).mean())


@pytest.mark.parametrize("C,heads", [(192, 8), (128, 8), (64, 4)])
def test_single_products_are_exact_to_a_rounding(C, heads):
    """Sets of one voxel and one weight per row: an output is a product of a product.  Each is off by 0.9 x 2^-24 (partial
    products that are not formed) and one rounding of 2^-24, and 0.1 x 2^-24 of truncations: 4 x 2^-24 for both."""
    from paper_2301_06051_b200 import api

    n = 2000
    rng = np.random.default_rng(C)
    case = di.random_case(C, n, (60, 60, 1), (1, 1, 1), 36, C, heads, 0)
    layer = case["blocks"][0][0]
    col, val = {}, {}
    for k in ("W_qkv", "W_o"):
        rows = layer[k].shape[0]
        col[k], val[k] = rng.integers(0, C, rows), rng.standard_normal(rows).astype(np.float32)
        layer[k] = np.zeros((rows, C), np.float32)
        layer[k][np.arange(rows), col[k]] = val[k]
        layer["b" + k[1:]] = np.zeros(rows, np.float32)
    ctx = api.Context(n, 3600, C)
    x = dev(case["feats"])
    table = ctx.partition(dev(case["coords"]), 1, case["grid"], case["window"], 36, 0)
    y = torch.empty_like(x)
    ctx.set_attention(x, table, api.device_weights(layer, api.FP32, ctx.device), y)
    assert ctx.status_sync() == 0
    v = case["feats"].astype(np.float64)[:, col["W_qkv"][2 * C :]] * val["W_qkv"][2 * C :]
    want = v[:, col["W_o"]] * val["W_o"]
    rel = np.abs(y.cpu().numpy() - want) / np.abs(want)
    assert rel.max() <= 4 * 2.0 ** -24, rel.max() * 2 ** 24


@pytest.mark.parametrize("C,heads,hidden,passes", [(128, 8, 0, 1), (192, 8, 384, 1), (192, 8, 64, 2)])
@pytest.mark.parametrize("kind", ["two hundred rows too many", "one offset far too large"])
def test_rows_that_no_set_fills_reach_no_voxel(oracle, C, heads, hidden, passes, kind):
    """Caller-made row offsets with more room than any set can fill, in a context whose buffers hold an earlier call's voxel
    ids: the sets that the offsets spoil are skipped, all other voxels come out right."""
    from paper_2301_06051_b200 import api

    tau, n = 36, 700 if passes == 1 else 14001
    grid = 48 if passes == 1 else 144
    case = di.random_case(C, n, (grid, grid, 1), (12, 12, 1), tau, C, heads, hidden, layernorm=hidden > 0)
    layer = case["blocks"][0][0]
    p = oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0)
    want = oracle.layer(case["feats"], p.set_table, layer)
    S = len(p.set_table)
    ctx = api.Context(n + (300 if passes == 2 else 0), (grid // 12) ** 2, C)
    x, w = dev(case["feats"]), api.device_weights(layer, api.FP32, ctx.device)
    table = upload_table(p.set_table)
    y = torch.full_like(x, 77.0)
    ctx.layer(x, table, w, y)  # (leaves its lists in the context)
    assert ctx.status_sync() == 0
    check_close(y.cpu().numpy(), want, "fp32", "sound offsets")
    at = S // 2 if passes == 1 else S // 4
    if kind == "one offset far too large":
        table.set_rowoff[at + 1] = 1 << 30
        spoiled = [at, at + 1]
    else:
        table.set_rowoff[at + 1 : S + 1] += 200
        spoiled = [at]
    y.fill_(77.0)
    ctx.layer(x, table, w, y)
    assert ctx.status_sync() == api.STATUS_BAD_INDEX
    got, members = y.cpu().numpy(), np.unique(p.set_table[spoiled])
    others = np.setdiff1d(np.arange(n), members)
    check_close(got[others], want[others], "fp32", "the other sets")
    assert np.all(got[members] == 77.0)


@pytest.mark.parametrize("tau,C,heads", [(36, 192, 8), (64, 192, 8), (96, 128, 4), (36, 64, 4)])
def test_bias_of_the_lowest_and_the_largest_float(oracle, tau, C, heads):
    """A position bias that is the lowest float for every pair of a head leaves its keys with equal weights, and so does one
    of the largest; sets of a single voxel, whose only pair is the zero offset, are among them."""
    from paper_2301_06051_b200 import api

    n = 400
    case = di.random_case(tau + C, n, (120, 36, 1), (12, 12, 1), tau, C, heads, 0)
    case["coords"][:, 1] = np.where(np.arange(n) < n - 4, case["coords"][:, 1] % 60, 60 + 12 * (np.arange(n) % 5))
    case["coords"] = case["coords"][np.sort(np.unique(case["coords"], axis=0, return_index=True)[1])]
    n = len(case["coords"])
    layer = case["blocks"][0][0]
    rng = np.random.default_rng(C)
    fmax = np.finfo(np.float32).max
    rpb = rng.standard_normal((heads, 23 * 23)).astype(np.float32)
    rpb[0], rpb[1] = -fmax, fmax
    rpb[2, (23 * 23) // 2] = -fmax  # the voxel itself is masked: a set of one voxel has no other key
    rpb[3, ::2] = -fmax
    layer["rpb"], layer["rpb_extent"] = rpb, (12, 12, 1)
    ctx = api.Context(n, 30, C)
    coords, x = dev(case["coords"]), dev(case["feats"][:n])
    table = ctx.partition(coords, 1, case["grid"], case["window"], tau, 0)
    y = torch.empty_like(x)
    ctx.set_attention(x, table, api.device_weights(layer, api.FP32, ctx.device), y, coords=coords)
    assert ctx.status_sync() == 0
    p = oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0)
    assert np.min(np.diff(rowoff_of(p.set_table))) == 1
    want, _ = oracle.set_attention(case["feats"][:n], p.set_table, layer["W_qkv"], layer["b_qkv"], layer["W_o"], layer["b_o"],
                                   heads, rpb=rpb, coords=case["coords"], rpb_extent=(12, 12, 1))
    check_close(y.cpu().numpy(), want, "fp32", "bias")


def test_voxels_in_many_sets_take_the_general_kernel(oracle):
    """A table with more rows than there are voxels (every set eight times over): the sets past the workspace's passes run on
    the kernel for general shapes, with the same results."""
    from paper_2301_06051_b200 import api

    n, tau, C, heads, hidden = 300, 36, 128, 8, 256
    case = di.random_case(7, n, (36, 36, 1), (12, 12, 1), tau, C, heads, hidden, layernorm=True)
    layer = case["blocks"][0][0]
    p = oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0)
    table = np.concatenate([p.set_table] * 8)
    ctx = api.Context(n, 9, C)
    x = dev(case["feats"])
    y = torch.empty_like(x)
    ctx.layer(x, upload_table(table), api.device_weights(layer, api.FP32, ctx.device), y)
    assert ctx.status_sync() == 0
    check_close(y.cpu().numpy(), oracle.layer(case["feats"], p.set_table, layer), "fp32", "voxels in many sets")


def test_passes_follow_the_call_and_not_the_context(oracle):
    """7,000 voxels (a pass of 192 channels holds 12,800) in contexts made for more: as many kernels and the same results as
    in a context of their size; 14,001 voxels take two passes in either."""
    from paper_2301_06051_b200 import api

    tau, C, heads = 36, 192, 8
    for n, sizes in ((7000, (7000, 12801, 40000)), (14001, (14001, 60000))):
        case = di.random_case(n, n, (144, 144, 1), (12, 12, 1), tau, C, heads, 64, layernorm=True)
        seen = []
        for size in sizes:
            ctx = api.Context(size, 144, C)
            x = dev(case["feats"])
            table = ctx.partition(dev(case["coords"]), 1, case["grid"], case["window"], tau, 0)
            w = api.device_weights(case["blocks"][0][0], api.FP32, ctx.device)
            y, before = torch.empty_like(x), ctx.launch_count()
            ctx.layer(x, table, w, y)
            assert ctx.status_sync() == 0
            seen.append((ctx.launch_count() - before, y))
        assert all(k == seen[0][0] and torch.equal(y, seen[0][1]) for k, y in seen)
        p = oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, 0)
        check_close(seen[0][1].cpu().numpy(), oracle.layer(case["feats"], p.set_table, case["blocks"][0][0]), "fp32", "n=%d" % n)


@pytest.mark.parametrize("C,heads,window,tau,hidden,option", [
    (192, 8, 12, 36, 384, "pe"),
    (192, 8, 2, 36, 0, ""),       # dozens of sets in a tile of 128 rows
    (128, 4, 30, 90, 256, "rpb"),
    (64, 4, 12, 36, 128, ""),
])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 3.4e38])
def test_a_wild_row_stays_in_its_set_in_fp32(C, heads, window, tau, hidden, option, value):
    """Voxels of features that are not finite, or whose products overflow, change no row outside their own sets (bitwise),
    although sets share tiles and the workspace keeps what they left."""
    from paper_2301_06051_b200 import api

    n, grid = 2500, (60, 60, 1)
    case = di.random_case(n + C, n, grid, (window, window, 1), tau, C, heads, hidden, layernorm=hidden > 0)
    layer, rng = case["blocks"][0][0], np.random.default_rng(C)
    if option == "rpb":
        layer["rpb"] = rng.standard_normal((heads, (2 * window - 1) ** 2)).astype(np.float32)
        layer["rpb_extent"] = (window, window, 1)
    ctx = api.Context(n, (60 // window) ** 2, C)
    coords, x = dev(case["coords"]), dev(case["feats"])
    pe = dev(rng.standard_normal((n, C)).astype(np.float32)) if option == "pe" else None
    t = ctx.partition(coords, 1, grid, (window, window, 1), tau, 0)
    w = api.device_weights(layer, api.FP32, ctx.device)
    clean, y = torch.empty_like(x), torch.empty_like(x)
    ctx.layer(x, t, w, clean, pe=pe, coords=coords)
    table = t.set_table[: int(t.num_sets.item())]
    wild = torch.as_tensor(rng.choice(n, 6, replace=False), device="cuda")
    sets = torch.isin(table, wild.to(torch.int32)).any(dim=1)
    inside = torch.zeros(n, dtype=torch.bool, device="cuda")
    inside[table[sets].reshape(-1).long()] = True
    spoilt = x.clone()
    spoilt[wild, ::5] = value
    spoilt[wild[0]] = value  # (and one whole row)
    ctx.layer(spoilt, t, w, y, pe=pe, coords=coords)
    assert ctx.status_sync() == 0
    assert torch.equal(y[~inside], clean[~inside])
    if value != value:
        assert torch.isnan(y[inside]).any(dim=1).all()
    ctx.layer(x, t, w, y, pe=pe, coords=coords)
    assert torch.equal(y, clean)


class _ContextHead(ctypes.Structure):
    """The beginning of the library's context, up to the address of its device status words."""
    _fields_ = [("device", ctypes.c_int), ("stream", ctypes.c_void_p), ("max_voxels", ctypes.c_int64), ("max_windows", ctypes.c_int64),
                ("max_channels", ctypes.c_int32), ("sm_count", ctypes.c_int), ("layer_ctas", ctypes.c_int), ("last_cuda_error", ctypes.c_int),
                ("attr_flags", ctypes.c_uint), ("launches", ctypes.c_int64), ("arena", ctypes.c_void_p), ("arena_bytes", ctypes.c_size_t),
                ("status", ctypes.c_void_p)]


def _status_words(ctx):
    head = _ContextHead.from_address(ctx._h.value)
    assert head.max_voxels == ctx.limits[0] and head.status == head.arena  # (the layout is still this one)

    class Words:
        __cuda_array_interface__ = {"shape": (3,), "typestr": "<i4", "data": (head.status, False), "version": 3}

    return torch.as_tensor(Words(), device="cuda")


@pytest.mark.parametrize("C,heads,hidden,copies", [(192, 8, 384, 1), (128, 8, 0, 1), (64, 4, 128, 6)])
def test_after_a_wait_has_given_up_the_call_leaves_y_alone(oracle, C, heads, hidden, copies):
    """The call's number is put down as that of a call one of whose waits has given up, as the kernel that gives up does: the
    kernels behind it store nothing to y, those for sets past the passes (voxels in several sets) included, and the next call is as ever."""
    from paper_2301_06051_b200 import api

    n, tau = 900, 36
    case = di.random_case(n + C, n, (48, 48, 1), (12, 12, 1), tau, C, heads, hidden, layernorm=hidden > 0)
    ctx = api.Context(n, 16, C)
    x = dev(case["feats"])
    p = [oracle.partition(case["coords"], 1, case["grid"], case["window"], tau, a).set_table for a in (0, 1)]
    tables = [upload_table(np.concatenate([q] * copies)) for q in p]
    layers = (case["blocks"][0] * 2)[: 1 if copies > 1 else 3]
    w = [api.device_weights(l, api.FP32, ctx.device) for l in layers]
    t = [tables[i & 1] for i in range(len(layers))]
    want = case["feats"]
    for i, l in enumerate(layers):
        want = oracle.layer(want, p[i & 1], l)
    y = torch.empty_like(x)
    words = _status_words(ctx)
    for given_up in (False, True, False):
        y.fill_(77.0)
        if given_up:
            words[2] = words[1] + 1
        ctx.layers(x, t, w, y)
        if given_up:
            assert torch.all(y == 77.0)
        else:
            check_close(y.cpu().numpy(), want, "fp32", "a call in which no wait gave up")
        assert ctx.status_sync() == 0


def test_chain_of_fp32_layers_on_several_tables(oracle):
    """Layers in one call share row lists and prepared weights, two at a time: five layers on three tables."""
    from paper_2301_06051_b200 import api

    n, tau, C, heads = 900, 36, 64, 4
    case = di.random_case(11, n, (48, 48, 1), (12, 12, 1), tau, C, heads, 128, layernorm=True)
    rng = np.random.default_rng(11)
    layers = [di.make_layer(rng, C, heads, 128, True, False) for _ in range(5)]
    ctx = api.Context(n, 16, C)
    coords, x = dev(case["coords"]), dev(case["feats"])
    t = [ctx.partition(coords, 1, case["grid"], w, tau, a) for w, a in (((12, 12, 1), 0), ((12, 12, 1), 1), ((16, 16, 1), 0))]
    r = [oracle.partition(case["coords"], 1, case["grid"], w, tau, a).set_table
         for w, a in (((12, 12, 1), 0), ((12, 12, 1), 1), ((16, 16, 1), 0))]
    order = [0, 1, 2, 2, 0]
    y = torch.empty_like(x)
    ctx.layers(x, [t[i] for i in order], [api.device_weights(l, api.FP32, ctx.device) for l in layers], y)
    assert ctx.status_sync() == 0
    want = case["feats"].astype(np.float64)
    for i, l in zip(order, layers):
        want = oracle.layer(want, r[i], l)
    check_close(y.cpu().numpy(), want, "fp32", "five layers")

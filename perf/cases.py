"""The performance cases of the DSVT library: what its users have it do, through the public entry points.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)` one more of the same ranges,
`prepare(case, seed)` what a program holds before the call (inputs, weights, the context or backbone), `run(state)` one
pass, `work(case)` the bytes and operations the pass cannot do without and `tolerance(case)` how far two correct
implementations of the same precision may lie apart.

Kinds of a case ("kind"):
  backbone  pipeline.Backbone.forward: both rotated partitions, the blocks, and with "pool" the attention-style pooling,
            the second stage and the projection to the bird's-eye-view map.  "hybrid": consecutive blocks alternate between (12, 12) windows and (24, 24) windows
            displaced by half, every layer with a relative position bias.
  block     dsvt_partition_rotated + dsvt_layers, the calls of a program that brings its own positional encoding.
  stages    pipeline.StagedBackbone.forward: the voxel variant's four stages with pooling along z between them, and the
            projection to the map.
  tables    dsvt_partition_rotated with the sorted order and the window arrays as further results.
  bev       dsvt_bev_scatter.
  stream    pipeline.FrameStream: frames from pinned host memory, results back to pinned host memory.
"""
import math

import numpy as np
import torch

import dsvt_inputs
from dsvt_inputs import configs
from paper_2301_06051_b200 import api, pipeline


def _case(kind, shape, n, **kw):
    c = dict(kind=kind, shape=shape, n=n, batch=1, grid=468, depth=1, window=12, set_size=36, C=192, heads=8, hidden=384,
             blocks=4, precision="bf16", pool=False, hybrid=False, pe=False, channels_last=False, frames=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a block of attention-only layers in fp32 on a few thousand pillars, latency counts
        dict(_case("backbone", "uniform", 2000, grid=64, C=128, hidden=0, blocks=1, precision="fp32"), name="tiny_fp32_block"),
        # a sparse near-field crop in bf16, one block with a learned positional term on queries and keys
        dict(_case("block", "pillar", 2531, blocks=1, pe=True), name="small_block_pe"),
        # full layers in fp32: the precision that exports and regression runs are checked at
        dict(_case("backbone", "pillar", 12345, blocks=1, precision="fp32"), name="fp32_block"),
        # the ordinary call: a pillar frame of 150 m x 150 m through a four-block backbone (the benchmark's workload)
        dict(_case("backbone", "pillar", 32000), name="pillar_frame"),
        # the nuScenes shapes: windows of 30 x 30, sets of 90, 128 channels
        dict(_case("backbone", "pillar", 30000, grid=360, window=30, set_size=90, C=128, hidden=256), name="wide_window_frame"),
        # hybrid windows with a relative position bias on every layer; a ragged count
        dict(_case("backbone", "pillar", 20011, blocks=2, hybrid=True), name="hybrid_bias_frame"),
        # the voxel variant on one stage: many voxels per window, full sets
        dict(_case("backbone", "voxel", 120000, depth=32), name="voxel_frame"),
        # the voxel variant's stage layout: one block per stage, pooling along z in between
        dict(_case("stages", "voxel", 120000, depth=32, set_size=48, blocks=1), name="voxel_stages"),
        # the largest: skewed occupancy, two blocks, 2 x 2 pooling, two blocks at half resolution
        dict(_case("backbone", "skew", 200000, grid=936, blocks=2, pool=True), name="skewed_pooled_frame"),
        # set tables only (for a caller with an attention of its own): four frames in one batch
        dict(_case("tables", "pillar", 128000, batch=4, blocks=0), name="tables_batch"),
        # the backbone's features onto the map that a 2-D network reads
        dict(_case("bev", "pillar", 32000, blocks=0), name="bev_map"),
        # six frames of differing size from the host and back: what a running sensor pipeline does
        dict(_case("stream", "pillar", 32000, frames=6), name="host_frame_stream"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["block_fp32", "block_pe", "pillar", "pillar", "wide", "hybrid", "voxel", "stages", "skew",
                         "tables", "bev", "stream"])
    if family == "block_fp32":
        full = rng.random() < 0.5
        return _case("backbone", "pillar" if full else "uniform", _log_uniform(rng, 1000, 12300 if full else 3500),
                     grid=468 if full else 64, C=rng.choice([128, 192]) if full else 128, hidden=0, blocks=1,
                     precision="fp32") | ({"hidden": 256} if full and rng.random() < 0.3 else {})
    if family == "block_pe":
        return _case("block", "pillar", _log_uniform(rng, 1500, 36000), blocks=rng.randint(1, 3), pe=rng.random() < 0.7)
    if family == "pillar":
        batch = rng.choice([1, 1, 2, 4])
        return _case("backbone", "pillar", batch * _log_uniform(rng, 1500, 36000), batch=batch, blocks=rng.randint(1, 4))
    if family == "wide":
        return _case("backbone", "pillar", _log_uniform(rng, 3000, 36000), grid=360, window=30, set_size=90, C=128,
                     hidden=256, blocks=rng.randint(1, 4))
    if family == "hybrid":
        return _case("backbone", "pillar", _log_uniform(rng, 3000, 36000), blocks=rng.randint(2, 4), hybrid=True)
    if family == "voxel":
        return _case("backbone", "voxel", _log_uniform(rng, 8000, 120000), depth=32, blocks=rng.randint(1, 4))
    if family == "stages":
        return _case("stages", "voxel", _log_uniform(rng, 12000, 120000), depth=32, set_size=48, blocks=1)
    if family == "skew":
        grid = 12 * rng.randint(30, 78)
        return _case("backbone", "skew", int(200000 * (grid / 936) ** 2 * rng.uniform(0.6, 1.0)), grid=grid, blocks=2, pool=True)
    if family == "tables":
        if rng.random() < 0.5:
            return _case("tables", "voxel", _log_uniform(rng, 5000, 120000), depth=32, blocks=0)
        batch = rng.choice([1, 2, 4])
        return _case("tables", "pillar", batch * _log_uniform(rng, 1500, 36000), batch=batch, blocks=0)
    if family == "bev":
        return _case("bev", "pillar", _log_uniform(rng, 3000, 36000), blocks=0, C=rng.choice([128, 192]),
                     grid=rng.choice([360, 468]), channels_last=rng.random() < 0.4)
    return _case("stream", "pillar", _log_uniform(rng, 8000, 36000), blocks=rng.randint(2, 4), frames=rng.randint(4, 7))


# ---------------------------------------------------------------------------------------------------------------
def _grid(case):
    return (case["grid"], case["grid"], case["depth"])


def _window(case):
    return (case["window"], case["window"], case["depth"])


def _coords(case, rng, n, batch):
    """int32 [n][4] = (b, x, y, z): distinct cells in arbitrary order, frame after frame."""
    out = []
    for b in range(batch):
        m = n // batch + (1 if b < n % batch else 0)
        if case["shape"] == "uniform":
            c = configs.unique_cells(rng, m, _grid(case))[:, 1:]
        elif case["shape"] == "voxel":
            c = configs.lidar_voxels(rng, m, case["grid"], case["depth"])
        elif case["shape"] == "skew":
            c = configs.skewed_pillars(rng, m, case["grid"], case["window"])
        else:
            c = configs.lidar_pillars(rng, m, case["grid"], 54.0 if case["grid"] == 360 else configs.HALF_RANGE,
                                      0.3 if case["grid"] == 360 else configs.CELL)
        out.append(np.concatenate([np.full((m, 1), b), c, np.zeros((m, 3 - c.shape[1]))], axis=1).astype(np.int32))
    return np.concatenate(out)


def _blocks(case, rng, count):
    bf16 = case["precision"] == "bf16"
    out = [[dsvt_inputs.make_layer(rng, case["C"], case["heads"], case["hidden"], case["hidden"] > 0, bf16)
            for _ in range(2)] for _ in range(count)]
    if case["hybrid"]:
        for i, blk in enumerate(out):
            ext = (12, 12, 1) if i % 2 == 0 else (24, 24, 1)
            for layer in blk:
                layer["rpb"] = (0.2 * rng.standard_normal((case["heads"], (2 * ext[0] - 1) * (2 * ext[1] - 1)))).astype(np.float32)
                layer["rpb_extent"] = ext
    return out


def _features(n, C, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn((n, C), generator=g, device="cuda")  # post-LayerNorm features: unit variance


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    n, C, kind, batch = case["n"], case["C"], case["kind"], case["batch"]
    bf16 = case["precision"] == "bf16"
    if kind == "stream":
        return _prepare_stream(case, rng, seed)
    coords = torch.from_numpy(_coords(case, rng, n, batch)).cuda()
    st = {"case": case, "coords": coords}
    if kind == "tables":
        w = _window(case)
        nw = batch * math.ceil(case["grid"] / w[0]) * math.ceil(case["grid"] / w[1])
        st["ctx"] = api.Context(n, nw, C)
        z = lambda *s: torch.zeros(s, dtype=torch.int32, device="cuda")
        st["tables"] = [api.SetTable(z(n, case["set_size"]), z(1), z(4 * n + 4), n, case["set_size"], z(n)) for _ in range(2)]
        t = st["tables"][0]
        t.win_start, t.win_count, t.win_setoff = z(nw + 1), z(nw), z(nw + 1)
        return st
    st["x"] = x = _features(n, C, seed)
    if kind == "bev":
        st["ctx"] = api.Context(n, 1, C)
        shape = (batch, case["grid"], case["grid"], C) if case["channels_last"] else (batch, C, case["grid"], case["grid"])
        st["map"] = torch.empty(shape, device="cuda")
        return st
    st["y"] = torch.empty_like(x)
    cfg = dict(n=n, batch=batch, grid=_grid(case), window=_window(case), set_size=case["set_size"], C=C,
               precision=case["precision"], blocks=_blocks(case, rng, case["blocks"]))
    if kind == "block":
        w = _window(case)
        st["ctx"] = api.Context(n, batch * math.ceil(case["grid"] / w[0]) * math.ceil(case["grid"] / w[1]), C)
        st["weights"] = [api.device_weights(l, api.BF16_FP32ACC, st["ctx"].device) for b in cfg["blocks"] for l in b]
        z = lambda *s: torch.zeros(s, dtype=torch.int32, device="cuda")
        st["tables"] = [api.SetTable(z(n, case["set_size"]), z(1), z(4 * n + 4), n, case["set_size"]) for _ in range(2)]
        st["pe"] = 0.3 * _features(n, C, seed + 1) if case["pe"] else None
        return st
    if kind == "stages":
        cfg["stages"], cfg["pools"] = [], []
        for z in (32, 8, 2, 1):
            cfg["stages"].append({"window": (12, 12, z), "blocks": _blocks(case, rng, 1)})
        for stride in (4, 4, 2):
            cfg["pools"].append({"shape": (1, 1, stride), "weights": dsvt_inputs.make_pool_weights(rng, C, case["heads"], bf16)})
        st["net"] = pipeline.StagedBackbone(cfg)
        st["map"] = torch.empty((batch, C, case["grid"], case["grid"]), device="cuda")
        return st
    if case["hybrid"]:
        cfg["block_windows"] = [((12, 12, 1), None) if i % 2 == 0 else ((24, 24, 1), (12, 12, 0)) for i in range(case["blocks"])]
    if case["pool"]:
        cfg["pool_shape"] = (2, 2, 1)
        cfg["pool"] = dsvt_inputs.make_pool_weights(rng, C, case["heads"], bf16)
        cfg["blocks_after_pool"] = _blocks(case, rng, case["blocks"])
        st["map"] = torch.empty((batch, C, case["grid"] // 2, case["grid"] // 2), device="cuda")
    st["net"] = pipeline.Backbone(cfg)
    return st


def _prepare_stream(case, rng, seed):
    n, C = case["n"], case["C"]
    cfg = dict(n=n, batch=1, grid=_grid(case), window=_window(case), set_size=case["set_size"], C=C,
               precision=case["precision"], blocks=_blocks(case, rng, case["blocks"]))
    net = pipeline.Backbone(cfg)
    frames = []
    for k in range(case["frames"]):  # a sensor's frames differ in size: the first holds n pillars, the others fewer
        m = n - k * n // 31
        c = torch.from_numpy(_coords(case, rng, m, 1)).pin_memory()
        f = torch.empty((m, C), pin_memory=True)
        f.copy_(_features(m, C, seed * 64 + k))
        frames.append((c, f, torch.zeros((m, C), pin_memory=True)))
    stream = pipeline.FrameStream(net.stage1, n, C, depth=4, lanes=2, layer_ctas=98)
    return {"case": case, "net": net, "stream": stream, "frames": frames}


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "stream":
        for c, f, out in st["frames"]:
            st["stream"].submit(c, f, out)
        st["stream"].wait()
        return [out for _, _, out in st["frames"]]
    if kind == "tables":
        t0, t1 = st["ctx"].partition_rotated(st["coords"], case["batch"], _grid(case), _window(case), case["set_size"],
                                             out=st["tables"])
        # (behind the row offsets, set_rowoff carries the library's own hand-over to its layer kernel)
        rows = case["n"] + 1
        return [t0.set_table, t1.set_table, t0.num_sets, t1.num_sets, t0.set_rowoff[:rows], t1.set_rowoff[:rows],
                t0.perm, t1.perm, t0.win_start, t0.win_count, t0.win_setoff]
    if kind == "bev":
        return st["ctx"].bev_scatter(st["coords"], st["x"], case["batch"], _grid(case), case["channels_last"], st["map"])
    if kind == "block":
        t = st["ctx"].partition_rotated(st["coords"], case["batch"], _grid(case), _window(case), case["set_size"],
                                        out=st["tables"])
        return st["ctx"].layers(st["x"], list(t) * case["blocks"], st["weights"], st["y"], pe=st["pe"])
    if kind == "stages":
        coords, feats = st["net"].forward(st["coords"], st["x"])
        return st["net"].ctx.bev_scatter(coords, feats, case["batch"], st["net"].grids[-1], out=st["map"])
    coords, feats, _ = st["net"].forward(st["coords"], st["x"], st["y"])
    if case["pool"]:
        return st["net"].ctx.bev_scatter(coords, feats, case["batch"], st["net"].pooled_grid, out=st["map"])
    return feats


# ---------------------------------------------------------------------------------------------------------------
def _layers_work(case, n, layers):
    """flops, weight bytes: projections and MLP per voxel, attention over the distinct members of a set (about 0.6
    of the slots are distinct members in these frames)."""
    C, h = case["C"], case["hidden"]
    wb = 2 if case["precision"] == "bf16" else 4
    return layers * n * (8.0 * C * C + 4.0 * C * h + 4.0 * C * 0.6 * case["set_size"]), layers * wb * (4.0 * C * C + 2.0 * C * h)


def _map_bytes(case, side):
    return 4.0 * case["batch"] * case["C"] * side * side


def work(case):
    n, C, kind = case["n"], case["C"], case["kind"]
    coords, rows = 16.0 * n, 4.0 * n * C
    if kind == "tables":  # coords in; per axis the table (about 0.6 of its slots distinct), sorted order and row offsets
        sets = n / (0.6 * case["set_size"])
        return {"bytes": coords + 2 * (4 * case["set_size"] * sets + 4 * n + 4 * sets), "flops": 0.0}
    if kind == "bev":
        return {"bytes": coords + rows + _map_bytes(case, case["grid"]), "flops": 0.0}
    layers = 2 * case["blocks"]
    if kind == "stream":
        f, w = _layers_work(case, 0.9 * n, layers)
        return {"bytes": case["frames"] * (0.9 * (coords + 2 * rows) + w), "flops": case["frames"] * f}
    if kind == "stages":  # (the first pooling halves the voxel count, the later ones change it little)
        (f, w), (f1, w1) = _layers_work(case, n, 2), _layers_work(case, n // 2, 6)
        pools = 8.0 * C * C * (n + n // 2 + n // 2)
        return {"bytes": coords + 1.5 * rows + w + w1 + 24.0 * C * C + _map_bytes(case, case["grid"]), "flops": f + f1 + pools}
    f, w = _layers_work(case, n, layers)
    by = coords + 2 * rows + w + (rows if case["pe"] else 0)
    if case["pool"]:  # about 0.4 n pooled voxels in these frames; queries and outputs per region, keys and values per voxel
        m = 0.4 * n
        f1, w1 = _layers_work(case, m, layers)
        return {"bytes": by - 0.6 * rows + w1 + 8.0 * C * C + _map_bytes(case, case["grid"] // 2), "flops": f + f1 + 4.0 * C * C * (m + n)}
    return {"bytes": by, "flops": f}


def tolerance(case):
    """Relative error (2-norm) and largest difference; four times what this library shows against the float64 oracle:
    fp32 4.5e-7 and 2.8e-6 (one block of full layers), bf16 3.0e-3 ... 4.2e-3 and up to 3.5e-2 (two to eight layers)."""
    if case["kind"] in ("tables", "bev"):
        return "exact"  # whole numbers; copied values
    if case["precision"] == "fp32":
        return {"rel": 2e-6, "max": 1.2e-5, "differ": 0.0}
    return {"rel": 1.6e-2, "max": 0.14, "differ": 0.0}

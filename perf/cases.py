"""What this library is used for, as timed cases: dense tensors sketched in every number format,
streams of boxes and CP terms, a server's mixed slices, tensors already in tree format, and the
recovery of the cores.  A case is a dict of plain values; `prepare` makes a user's inputs and plan on
the GPU, `run` is one pass through the public entry points, `exact` is the same result from the
definitions in 64 bits (per-mode Gaussian factors, Khatri-Rao blocks rounded once to the sketch
format, one contraction per tree node)."""
import functools
import math

import numpy as np
import torch

from paper_2412_06111_gb300 import api

FORMATS = {"f64": api.F64, "f32": api.F32, "bf16": api.BF16, "bf16x2": api.BF16X2, "e4m3": api.E4M3}
STORED = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16,
          "bf16x2": torch.float32, "e4m3": torch.float32}
# rounding of the DRM factors and of the Khatri-Rao blocks of the first-level pass
DRM = {"f64": "f64", "f32": "f32", "bf16": "bf16", "bf16x2": "bf16", "e4m3": "e4m3"}
STREAM_UPDATES = 8      # updates a streaming pass folds in, one after another
SLICES = 4              # slices each served stream receives in a pass


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _dims(n, d):
    return "x".join([str(n)] * d)


def listed():
    return [
        # the smallest whole call: one 24^4 binary64 tensor sketched and its cores recovered (launches, latency)
        dict(name="f64_24p4_to_cores", kind="whole", fmt="f64", variant="ttnn", tree="binary", dims=_dims(24, 4), r=5, p=5),
        # a server with mixed resident streams (orders 3-6, modes 16-128, all trees), a burst of mode slices
        dict(name="serve_mix_16", kind="serve", fmt="bf16", streams=16, mix=7),
        # a 32^6 tensor that arrives as additive updates: a rank-2 CP term and a dense 32^3 box each
        dict(name="stream_tt_32p6", kind="stream", fmt="bf16", variant="ttnn", tree="tt", dims=_dims(32, 6), r=16, p=8, box=32, cp=2),
        # the flagship: a 64^5 grid function stored in bfloat16, one pass, binary tree
        dict(name="bf16_64p5", kind="dense", fmt="bf16", variant="ttnn", tree="binary", dims=_dims(64, 5), r=20, p=10),
        # mode sizes nobody chose for a machine: 45^5 in bfloat16, the sequential variant
        dict(name="sttnn_bf16_45p5", kind="dense", fmt="bf16", variant="sttnn", tree="binary", dims=_dims(45, 5), r=20, p=10),
        # the same grid function kept in binary32 and sketched in binary32
        dict(name="f32_64p5", kind="dense", fmt="f32", variant="ttnn", tree="binary", dims=_dims(64, 5), r=20, p=10),
        # a binary32 tensor that arrives in slabs of its first mode (a time step, one rank's share)
        dict(name="f32_slab_8x64p4", kind="slab", fmt="f32", variant="ttnn", tree="binary", dims=_dims(64, 5), r=20, p=10, slab=8),
        # binary32 storage, split in two bfloat16 products, at another size
        dict(name="bf16x2_48p5", kind="dense", fmt="bf16x2", variant="ttnn", tree="binary", dims=_dims(48, 5), r=16, p=8),
        # a binary32 tensor quantised to E4M3 tiles and sketched from them
        dict(name="e4m3_64p5_quantised", kind="dense", fmt="e4m3", variant="ttnn", tree="binary", dims=_dims(64, 5), r=20, p=10),
        # the Hilbert tensor 20^6 in binary64 on the six-mode example tree
        dict(name="f64_hilbert_20p6", kind="dense", fmt="f64", variant="ttnn", tree="toy", dims=_dims(20, 6), r=10, p=5),
        # rounding of a tensor in tree format: order 8, modes 64, edge ranks 200, to 30
        dict(name="ttn_o8_rank200", kind="ttn", fmt="bf16", variant="ttnn", tree="binary", dims=_dims(64, 8), r=30, p=15, rank=200),
        # recovery of the cores from resident sketches (QR, pseudo-inverse, assembly in binary64)
        dict(name="recover_64p5", kind="recover", fmt="bf16", variant="ttnn", tree="binary", dims=_dims(64, 5), r=20, p=10, decay=0.55),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_dims(rng, d, most, least, step=1, hi=512):
    """d mode sizes of at most `most` entries together (log-uniform between `least` and `most`), each
    within a factor of about two of the others and a multiple of `step`."""
    target = math.exp(rng.uniform(math.log(least), math.log(most)))
    mean = target ** (1.0 / d)
    dims = []
    for k in range(d):
        n = mean * math.exp(rng.uniform(-0.4, 0.4))
        dims.append(max(step, 4, min(hi, int(n) // step * step)))
    while math.prod(dims) > most:
        k = dims.index(max(dims))
        dims[k] -= step
    return dims


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "dense", "slab", "stream", "serve", "ttn", "recover", "whole"])
    if kind == "serve":
        return dict(kind=kind, fmt="bf16", streams=rng.randint(4, 20), mix=rng.randint(100, 10 ** 6))
    case = dict(kind=kind, fmt="bf16", variant="ttnn", tree="binary")
    d = rng.randint(3, 6)
    r = rng.randint(4, 32)
    if kind == "dense":
        case["fmt"] = rng.choice(["bf16", "bf16", "f32", "bf16x2", "e4m3", "f64"])
        if case["fmt"] in ("bf16", "f32", "f64"):
            case["variant"] = rng.choice(["ttnn", "ttnn", "sttnn"])
            if case["variant"] == "ttnn":
                case["tree"] = rng.choice(["binary", "binary", "tt", "tucker"])
        if case["fmt"] == "f64":
            dims, r = _draw_dims(rng, d, 4e7, 2e4), rng.randint(4, 12)
        elif case["fmt"] in ("bf16x2", "e4m3"):
            d = max(d, 4)
            dims = _draw_dims(rng, d, 5e8, 3e5, 16)
        elif rng.random() < 0.5:
            dims = _draw_dims(rng, d, 5e8, 3e5, 8)       # sizes that were chosen for alignment
        else:
            dims = _draw_dims(rng, d, 1.8e8, 1e5)        # sizes that were not
    elif kind == "slab":
        case["fmt"] = rng.choice(["bf16", "f32", "f32", "f64"])
        d = max(d, 4)
        dims = _draw_dims(rng, d, 1e7 if case["fmt"] == "f64" else 5e8, 1e5, rng.choice([1, 8]))
        case["slab"] = max(1, dims[0] // rng.randint(3, 10))
        r = min(r, 24)
    elif kind == "stream":
        case["tree"] = rng.choice(["tt", "tt", "binary", "tucker"])
        d = rng.randint(4, 6) if case["tree"] != "tucker" else 4
        n = rng.randint(16, 48)
        dims = [n] * d if n ** d <= 1.1e9 else [24] * d
        r = rng.randint(6, 20)
        case["box"], case["cp"] = rng.randint(8, min(dims)), rng.randint(1, 20)
    elif kind == "ttn":
        case["fmt"] = rng.choice(["bf16", "f32", "f64"])
        d = rng.randint(4, 8)
        case["rank"] = _log_int(rng, 24, 70 if case["fmt"] == "f64" else 180)
        dims = [_log_int(rng, 16, 500 if case["fmt"] == "f64" else 128) for _ in range(d)]
        r = rng.randint(6, max(7, min(32, case["rank"] // 3)))
    elif kind == "recover":
        case["fmt"] = rng.choice(["bf16", "f64"])
        case["decay"] = round(rng.uniform(0.5, 0.95), 3)
        r = rng.randint(4, 40) if case["decay"] > 0.7 else rng.randint(4, 16)
        dims = [rng.randint(20, 96) for _ in range(d)]
    else:
        case["fmt"] = "f64"
        dims = _draw_dims(rng, rng.randint(3, 5), 6e5, 2e4)
        r = rng.randint(3, 6)
    r = min(r, max(2, max(dims) // 2))      # the largest leaf at least is compressed
    case["dims"] = "x".join(str(n) for n in dims)
    case["r"], case["p"] = r, max(2, r // 2)
    return case


# ---------------------------------------------------------------------------
# trees and their nodes (row-major modes; nodes in level order, as the state lays them out)
# ---------------------------------------------------------------------------
def _tree(name, d):
    """(parent, leaf_modes, identity) of a balanced binary, tensor-train, Tucker or example tree."""
    def binary(lo, hi):
        if hi - lo == 1:
            return lo
        mid = lo + (hi - lo + 1) // 2
        return binary(lo, mid), binary(mid, hi)

    if name == "tt":
        spec = 0
        for k in range(1, d):
            spec = (spec, k)
    else:
        spec = {"binary": lambda: binary(0, d), "tucker": lambda: tuple(range(d)),
                "toy": lambda: (((0, 1), 2), 3, (4, 5))}[name]()
    parent, modes = [], []

    def add(s, p):
        v = len(parent)
        parent.append(p)
        modes.append([s] if isinstance(s, int) else [])
        if not isinstance(s, int):
            for c in s:
                add(c, v)

    add(spec, -1)
    return parent, modes, [name == "tt" and bool(m) and m[0] >= 1 for m in modes]


class Node:
    pass


class Layout:
    """Nodes of a case's tree with their ranks as the library clips them, and the first-level split."""

    def __init__(self, tree, dims, r, p, variant):
        self.tree, self.dims, self.variant = tree, dims, variant
        parent, modes, ident = tree
        self.nodes = [Node() for _ in parent]
        for v, nd in enumerate(self.nodes):
            nd.v, nd.parent, nd.ch, nd.modes = v, parent[v], [], list(modes[v])
        for v in reversed(range(len(parent))):      # children come after their parents
            if parent[v] >= 0:
                self.nodes[parent[v]].ch.insert(0, v)
                self.nodes[parent[v]].modes += self.nodes[v].modes
        total = math.prod(dims)
        for v, nd in enumerate(self.nodes):
            nd.modes = sorted(nd.modes)
            nd.lo, nd.hi = nd.modes[0], nd.modes[-1] + 1
            nd.leaf, nd.n = not nd.ch, math.prod(dims[nd.lo:nd.hi])
            nd.identity = nd.leaf and parent[v] >= 0 and (ident[v] or r >= nd.n)
            nd.r = nd.n if nd.identity else min(r, nd.n, total // nd.n)
            nd.s = nd.n if nd.identity else nd.r + min(p, nd.n - nd.r)
            nd.sketched = parent[v] >= 0 and not nd.identity
        self.order, level = [], [0]
        while level:
            self.order += level
            level = [c for v in level for c in self.nodes[v].ch]
        sk = [self.nodes[v] for v in self.order if self.nodes[v].sketched]
        self.rmax, self.smax = max(n.r for n in sk), max(n.s for n in sk)
        root = self.nodes[0].ch
        s = [self.nodes[c].s for c in root]
        if variant == "sttnn":
            a, self.ychild = 1, root[0]
        elif len(root) == 2:
            a, self.ychild = 1, root[1] if s[1] <= s[0] else root[0]
        else:
            a, self.ychild = len(root) - 1, root[-1]
        self.left = range(0, self.nodes[root[a - 1]].hi)
        self.right = range(self.left.stop, len(dims))

    def reuse(self, v):
        """Groups the sequential variant has contracted before node v: its and its ancestors' earlier siblings."""
        out, u = [], v
        while self.nodes[u].parent >= 0:
            for c in self.nodes[self.nodes[u].parent].ch:
                if c == u:
                    break
                if not self.nodes[c].identity:
                    out.append(c)
            u = self.nodes[u].parent
        return sorted(out, key=lambda c: self.nodes[c].lo)

    def psi_shape(self, nd):
        if nd.leaf:
            return [nd.n, nd.r]
        return [self.nodes[c].s for c in nd.ch] + ([nd.r] if nd.parent >= 0 else [])

    def state_elems(self):
        return sum(math.prod(self.psi_shape(n)) + (n.s * n.r if n.sketched else 0)
                   for n in self.nodes if n.sketched or n.parent < 0)

    def widths(self):
        """Columns the dense tensor is multiplied by: X of the left and right groups, Y of one root child."""
        sub = lambda g: max([n.r for n in self.nodes if n.sketched and n.lo in g and n.hi - 1 in g] + [0])
        return sub(self.left) + (sub(self.right) if self.variant == "ttnn" else 0) + self.nodes[self.ychild].s


def _layout(case):
    dims = [int(n) for n in case["dims"].split("x")]
    return Layout(_tree(case["tree"], len(dims)), dims, case["r"], case["p"], case["variant"])


def _mix(case):
    """The layouts of a server case: orders 3-6, modes 16-128, at most 2e8 entries, the three trees, r 4-32."""
    rng = np.random.default_rng(case["mix"])
    out = []
    while len(out) < case["streams"]:
        d = int(rng.integers(3, 7))
        dims = [int(n) for n in rng.choice([16, 32, 64, 128], size=d)]
        r = int(rng.integers(4, 33))
        tree = ("binary", "tt", "tucker")[int(rng.integers(0, 3))]
        if math.prod(dims) > 2e8:
            continue
        lay = Layout(_tree(tree, d), dims, r, r // 2, "ttnn")
        if lay.state_elems() <= 4_000_000:
            out.append((lay, r))
    return out


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _grid_function(dims, seed, dtype):
    """1 / (x_1 + ... + x_d) on grids x_mu = a + (0 .. 1) b with seeded a, b near 1 (a Hilbert-type tensor
    with a fast-decaying spectrum), in the storage format."""
    rng = np.random.default_rng(seed)
    s = torch.zeros([1] * len(dims), dtype=torch.float64, device="cuda")
    for mu, n in enumerate(dims):
        a, b = rng.uniform(0.8, 1.2, size=2)
        x = a + b * torch.arange(n, dtype=torch.float64, device="cuda") / max(n - 1, 1)
        s = s + x.reshape([-1 if k == mu else 1 for k in range(len(dims))])
    return s.reciprocal_().to(dtype)


def _low_rank_noise(lay, rank, seed):
    """A tensor of exact tree ranks `rank` plus Gaussian noise of 1e-8 of its norm."""
    g = _gen(seed)
    cores = []
    for nd in lay.nodes:
        up = [rank] if nd.parent >= 0 else []
        cores.append(torch.randn(up + ([nd.n] if nd.leaf else [rank] * len(nd.ch)), dtype=torch.float64, device="cuda", generator=g))

    def full(v):
        out = cores[v]
        for c in lay.nodes[v].ch:
            out = torch.tensordot(out, full(c), dims=([0 if lay.nodes[v].parent < 0 else 1], [0]))
        return out.reshape(([rank] if lay.nodes[v].parent >= 0 else []) + [-1])

    t = full(0).reshape(lay.dims)
    e = torch.randn(lay.dims, dtype=torch.float64, device="cuda", generator=g)
    return t + e * (1e-8 * t.norm() / e.norm())


def _stream_updates(case, lay, seed):
    """STREAM_UPDATES of (CP factors, box offset, box extent, box data): three modes of a box vary, the others are fixed."""
    rng, g, out = np.random.default_rng(seed), _gen(seed), []
    for _ in range(STREAM_UPDATES):
        off, ext = [int(rng.integers(0, n)) for n in lay.dims], [1] * len(lay.dims)
        for mu in rng.choice(len(lay.dims), size=3, replace=False):
            ext[mu] = min(case["box"], lay.dims[mu])
            off[mu] = int(rng.integers(0, lay.dims[mu] - ext[mu] + 1))
        box = (0.1 * torch.randn(ext, dtype=torch.float64, device="cuda", generator=g)).to(STORED[case["fmt"]])
        cp = [torch.randn((n, case["cp"]), dtype=torch.float64, device="cuda", generator=g) for n in lay.dims]
        out.append((cp, off, ext, box))
    return out


def _slices(case, mix, seed):
    """The served requests in submission order: (stream, offset, extent, slice data)."""
    rng, g, out = np.random.default_rng(seed), _gen(seed), []
    for _ in range(SLICES):
        for k, (lay, _) in enumerate(mix):
            mu = int(rng.integers(0, len(lay.dims)))
            off, ext = [0] * len(lay.dims), list(lay.dims)
            off[mu], ext[mu] = int(rng.integers(0, lay.dims[mu])), 1
            out.append((k, off, ext, torch.randn(ext, device="cuda", generator=g).to(torch.bfloat16)))
    return out


def _ttn_cores(lay, rank, seed):
    """Input cores: a direct sum of a dominant network (about a sixth of the rank) and a noise network of 1/100 of its norm."""
    g, lead = _gen(seed), max(2, rank * 3 // 20)
    edges = len(lay.nodes) - 1
    cores = []
    for nd in lay.nodes:
        shape = ([rank] if nd.parent >= 0 else []) + ([nd.n] if nd.leaf else [rank] * len(nd.ch))
        core = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for lo, k, norm in ((0, lead, 100.0), (lead, rank - lead, 1.0)):
            part = [k if i < len(shape) and not (nd.leaf and i == len(shape) - 1) else n for i, n in enumerate(shape)]
            x = torch.randn(part, dtype=torch.float64, device="cuda", generator=g) / math.sqrt(rank)
            if nd.parent < 0:   # the expected norm of the part's network is `norm`
                x *= norm / math.sqrt(float(k) ** edges * float(rank) ** -len(lay.nodes) * math.prod(lay.dims))
            core[tuple(slice(0, n) if nd.leaf and i == len(shape) - 1 else slice(lo, lo + k) for i, n in enumerate(shape))] = x
        cores.append(core.contiguous())
    return cores


def _cp_decaying(lay, decay, seed):
    """Factors and weights of a CP tensor with geometric weights: what a decaying spectrum leaves in the sketches."""
    g, k = _gen(seed), lay.smax + 8
    w = torch.tensor([max(decay ** q, 1e-7) for q in range(k)], dtype=torch.float64, device="cuda")
    return w, [torch.randn((n, k), dtype=torch.float64, device="cuda", generator=g) / math.sqrt(n) for n in lay.dims]


def _box_tensor(case, lay, seed):
    """(data in storage format, offset, extent); offset None for whole tensors."""
    if case["kind"] == "slab":
        rng = np.random.default_rng(seed)
        off, ext = [0] * len(lay.dims), list(lay.dims)
        ext[0], off[0] = case["slab"], int(rng.integers(0, lay.dims[0] - case["slab"] + 1))
        return _grid_function(ext, seed, STORED[case["fmt"]]), off, ext
    if case["kind"] == "whole":
        return _low_rank_noise(lay, case["r"], seed), None, None
    return _grid_function(lay.dims, seed, STORED[case["fmt"]]), None, None


# ---------------------------------------------------------------------------
# states: what a user's program holds before the call
# ---------------------------------------------------------------------------
class _Handles:
    """The library's handles of one state, freed when the last user of their buffers is gone."""
    plan = state = server = None

    def __del__(self):
        if self.server is not None:
            api.ttnn_server_destroy(self.server)
        if self.state is not None:
            api.ttnn_state_destroy(self.state)
        if self.plan is not None:
            api.ttnn_plan_destroy(self.plan)


class _Buffer:
    """A sketch state's device buffer, and what keeps it allocated."""

    def __init__(self, handles, state, fmt):
        ptr, n = api.ttnn_state_buffer(state)
        self.handles = handles
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f8" if fmt == "f64" else "<f4", "data": (ptr, False), "version": 3}


def _accumulators(handles, state, fmt):
    """The tensor over a sketch state's buffer; it keeps the state alive."""
    return torch.as_tensor(_Buffer(handles, state, fmt), device="cuda")


class State:
    """Inputs, handles and outputs of one case."""


def prepare(case, seed):
    st = State()
    st.case, h = case, _Handles()
    st.h = h
    if case["kind"] == "serve":
        mix = _mix(case)
        st.requests = _slices(case, mix, seed)
        h.server = api.ttnn_server_create(64 << 30, max_batch=64, queue_capacity=1024, workers=8)
        st.sids = [api.ttnn_server_open(h.server, lay.tree, lay.dims, [r] * len(lay.nodes), [r // 2] * len(lay.nodes),
                                        2024 + seed + k, sketch_dtype=api.BF16) for k, (lay, r) in enumerate(mix)]
        st.out = [_accumulators(h, api.ttnn_server_stream_state(h.server, s), "bf16") for s in st.sids]
        torch.cuda.synchronize()
        return st
    lay = _layout(case)
    n = len(lay.nodes)
    h.plan = api.ttnn_plan_create(lay.tree, lay.dims, [case["r"]] * n, [case["p"]] * n, 2024 + seed,
                                  variant=api.VARIANT_STTNN if case["variant"] == "sttnn" else api.VARIANT_TTNN,
                                  sketch_dtype=FORMATS[case["fmt"]],
                                  flags=api.FLAG_STRUCTURED_ONLY if case["kind"] == "ttn" else 0)
    h.state = api.ttnn_state_create(h.plan)
    st.out = _accumulators(h, h.state, case["fmt"])
    st.cores = torch.zeros(api.ttnn_plan_sizes(h.plan)[2], dtype=torch.float64, device="cuda")
    if case["kind"] in ("dense", "slab", "whole"):
        st.data, st.off, st.ext = _box_tensor(case, lay, seed)
        if case["fmt"] == "e4m3":
            rows = math.prod(lay.dims[:lay.left.stop])
            tiles = -(-rows // 128) * -(-(st.data.numel() // rows) // 128)
            st.q8 = torch.empty(st.data.numel(), dtype=torch.uint8, device="cuda")
            st.scales = torch.empty(tiles, dtype=torch.float32, device="cuda")
    elif case["kind"] == "stream":
        st.updates = _stream_updates(case, lay, seed)
        st.weights = [1.0] * case["cp"]
    elif case["kind"] == "ttn":
        st.inputs, st.ranks = _ttn_cores(lay, case["rank"], seed), [case["rank"]] * n
    elif case["kind"] == "recover":
        w, a = _cp_decaying(lay, case["decay"], seed)
        acc = _flat(lay, *_sketch_cp(lay, _Drm(lay, 2024 + seed, DRM[case["fmt"]], False), w, a))
        api.ttnn_state_load(h.state, acc.to(st.out.dtype).cpu().numpy())
    torch.cuda.synchronize()
    return st


def run(st):
    kind, h = st.case["kind"], st.h
    if kind == "serve":
        tickets = [api.ttnn_server_submit(h.server, st.sids[k], data, off, ext) for k, off, ext, data in st.requests]
        for t in tickets:
            if api.ttnn_server_wait(h.server, t, 60_000_000) != 0:
                raise RuntimeError(api.last_error_message())
        return st.out
    if kind == "stream":
        for cp, off, ext, box in st.updates:
            api.ttnn_update_cp(h.state, st.weights, cp)
            api.ttnn_update_dense(h.state, box, off, ext)
        return st.out
    if kind == "recover":
        api.ttnn_recover(h.state, st.cores)
        return st.cores
    api.ttnn_state_zero(h.state)
    if kind == "ttn":
        api.ttnn_update_ttn(h.state, st.inputs, st.ranks)
        return st.out
    if st.case["fmt"] == "e4m3":
        api.ttnn_fp8_quantize(h.plan, st.data, st.q8, st.scales)
        api.ttnn_update_dense(h.state, st.q8, tile_scale=st.scales)
        return {"q": st.q8, "scale": st.scales, "state": st.out}
    api.ttnn_update_dense(h.state, st.data, st.off, st.ext)
    if kind == "whole":
        api.ttnn_recover(h.state, st.cores)
        return {"state": st.out, "cores": st.cores}
    return st.out


def work(case):
    """Bytes: the tensor (or cores, or sketches) read once, the sketches (or cores) written once.
    Flops: the contractions that no split of the work avoids."""
    if case["kind"] == "serve":
        nbytes = flops = 0.0
        for lay, _ in _mix(case):
            entries = SLICES * sum(math.prod(lay.dims) / n for n in lay.dims) / len(lay.dims)   # mean over the sliced mode
            nbytes += 2 * entries + 4 * lay.state_elems()
            flops += 2 * entries * lay.widths()
        return {"bytes": nbytes, "flops": flops}
    lay = _layout(case)
    out = lay.state_elems() * (8 if case["fmt"] == "f64" else 4)
    if case["kind"] == "stream":
        box = STREAM_UPDATES * min(case["box"], min(lay.dims)) ** 3
        terms = STREAM_UPDATES * case["cp"]
        return {"bytes": 2 * box + 8 * terms * sum(lay.dims) + out, "flops": 2.0 * box * lay.widths() + 2.0 * terms * lay.state_elems()}
    if case["kind"] == "ttn":
        size = lambda nd: (case["rank"] if nd.parent >= 0 else 1) * (nd.n if nd.leaf else case["rank"] ** len(nd.ch))
        elems = sum(size(nd) for nd in lay.nodes)
        # each core against X and Y of its subtree (up) and against the environment (down)
        return {"bytes": 8 * elems + out, "flops": 2.0 * elems * (2 * lay.rmax + lay.smax)}
    if case["kind"] == "recover":
        cores = sum(nd.r * nd.n if nd.leaf else (nd.r if nd.parent >= 0 else 1) * math.prod(lay.nodes[c].r for c in nd.ch)
                    for nd in lay.nodes)
        return {"bytes": out + 8 * cores, "flops": sum(4.0 * nd.s * nd.r ** 2 + 2.0 * math.prod(lay.psi_shape(nd)) * nd.r for nd in lay.nodes if nd.sketched)}
    entries = math.prod(lay.dims) * (case["slab"] / lay.dims[0] if case["kind"] == "slab" else 1)
    stored = {"f64": 8, "f32": 4, "bf16": 2, "bf16x2": 4, "e4m3": 4 + 1 + 1}[case["fmt"]]   # E4M3: read, written, read again
    return {"bytes": stored * entries + out, "flops": 2.0 * entries * lay.widths()}


# ---------------------------------------------------------------------------
# the definitions in 64 bits
# ---------------------------------------------------------------------------
_SIGNIFICANT = {"bf16": 8, "e4m3": 4}


def _round(x, fmt):
    """Nearest-even rounding of binary64 values into a format (normal range; E4M3 with its subnormals, saturating)."""
    if fmt == "f64":
        return x
    if fmt == "f32":
        return x.float().double()
    e = torch.frexp(x)[1].long() - _SIGNIFICANT[fmt]
    if fmt == "e4m3":
        e = e.clamp(min=-9)
    q = ((e + 1023) << 52).view(torch.float64)      # 2^e
    y = torch.round(x / q) * q
    return y.clamp(-448.0, 448.0) if fmt == "e4m3" else y


def _gaussian(seed, kind, ident, rows, cols):
    """N(0,1) draws: Philox4x32-10 (Salmon et al. 2011) on counter (i, j // 2, kind << 24 | ident, 0), two 53-bit
    uniforms per call, Box-Muller."""
    m32 = np.uint64(0xFFFFFFFF)
    i, j = np.arange(rows, dtype=np.uint64)[:, None], np.arange(cols, dtype=np.uint64)[None, :]
    c = [i + np.uint64(0) * j, (j >> np.uint64(1)) + np.uint64(0) * i, np.full((rows, cols), (kind << 24) | ident, np.uint64),
         np.zeros((rows, cols), np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    top = lambda a, b: (((a << np.uint64(32)) | b) >> np.uint64(11)).astype(np.float64)
    u1, u2 = (top(c[0], c[1]) + 1.0) * 2.0 ** -53, top(c[2], c[3]) * 2.0 ** -53
    r, t = np.sqrt(-2.0 * np.log(u1)), 2.0 * np.pi * u2
    return torch.from_numpy(np.where(np.arange(cols) % 2 == 0, r * np.cos(t), r * np.sin(t))).cuda()


def _kr(mats):
    """Column-wise Khatri-Rao product, the first factor's row index slowest."""
    out = mats[0]
    for m in mats[1:]:
        out = (out[:, None, :] * m[None, :, :]).reshape(-1, out.shape[1])
    return out


class _Drm:
    """The per-mode factors of a plan and the blocks of its first-level pass.  blocks=False: the inputs are structured
    (CP, tree format) and no Khatri-Rao block is rounded a second time."""

    def __init__(self, lay, seed, fmt, blocks=True, lo=None, ext=None):
        dims = lay.dims
        rows = lambda m, mu: m if lo is None else m[lo[mu]:lo[mu] + ext[mu]]
        self.lay = lay
        self.X = [rows(_round(_gaussian(seed, 1, mu, n, lay.rmax), fmt), mu) for mu, n in enumerate(dims)]
        self.Y = [rows(_round(_gaussian(seed, 2, mu, n, lay.smax), fmt), mu) for mu, n in enumerate(dims)]
        self.XT = {v: _round(_gaussian(seed, 3, i, lay.nodes[v].s, lay.rmax), fmt)
                   for i, v in enumerate(lay.order) if lay.nodes[v].sketched}
        self.again = (lambda b: _round(b, fmt)) if blocks else (lambda b: b)
        self.eye = {nd.v: rows(torch.eye(nd.n, dtype=torch.float64, device="cuda"), nd.lo)
                    for nd in lay.nodes if nd.identity and nd.hi - nd.lo == 1}

    @functools.cached_property
    def BR(self):
        return self.again(_kr([self.X[mu] for mu in self.lay.right]))

    @functools.cached_property
    def BL(self):
        return self.again(_kr([self.X[mu] for mu in self.lay.left]))

    @functools.cached_property
    def Yside(self):
        y = self.lay.nodes[self.lay.ychild]
        return self.again(_kr(self.Y[y.lo:y.hi]))

    def Yt(self, v):
        nd = self.lay.nodes[v]
        if nd.identity:
            return self.eye[v]
        return self.Yside[:, :nd.s] if v == self.lay.ychild else _kr([self.Y[mu] for mu in range(nd.lo, nd.hi)])[:, :nd.s]

    def Xt(self, v, axes):
        """X over the axes ("m", mode) or ("g", contracted group) outside node v."""
        lay, nd = self.lay, self.lay.nodes[v]
        pick = lambda ax: self.XT[ax[1]] if ax[0] == "g" else self.X[ax[1]]
        inside = lambda ax, g: ax[0] == "m" and ax[1] in g
        rest = [ax for ax in axes if not inside(ax, range(nd.lo, nd.hi))]
        if nd.lo in lay.left:
            mats = [pick(ax) for ax in rest if not inside(ax, lay.right)] + [self.BR]
        elif lay.variant == "sttnn":
            mats = [pick(ax) for ax in rest]
        else:
            mats = [self.BL] + [pick(ax) for ax in rest if not inside(ax, lay.left)]
        return _kr([m[:, :nd.r] for m in mats])


def _on_axis(t, k, m):
    return torch.movedim(torch.tensordot(t, m, dims=([k], [0])), -1, k)


def _psi(lay, drm, nd, g, tail):
    p = g.reshape([drm.Yt(c).shape[0] for c in nd.ch] + tail)
    for k, c in enumerate(nd.ch):
        if not lay.nodes[c].identity or drm.Yt(c).shape[0] != lay.nodes[c].n:
            p = _on_axis(p, k, drm.Yt(c))
    return p


def _sketch_dense(lay, drm, t):
    """(Omega, Psi) of a dense binary64 tensor (or of a box, when the factors' rows are the box's)."""
    om, ps = {}, {}
    for nd in lay.nodes:
        if not nd.sketched:
            continue
        axes, u = [("m", mu) for mu in range(len(lay.dims))], t
        for s in lay.reuse(nd.v) if lay.variant == "sttnn" else []:
            k, g = axes.index(("m", lay.nodes[s].lo)), lay.nodes[s]
            u = _on_axis(u.reshape(u.shape[:k] + (-1,) + u.shape[k + g.hi - g.lo:]), k, drm.Yt(s))
            axes[k:k + g.hi - g.lo] = [("g", s)]
        k, m = axes.index(("m", nd.lo)), nd.hi - nd.lo
        rows, cols = math.prod(u.shape[k:k + m]), math.prod(u.shape[:k])
        x = drm.Xt(nd.v, axes).reshape(cols, -1, nd.r)      # the axes before the node, those after it
        g = torch.zeros((rows, nd.r), dtype=torch.float64, device="cuda")
        for a, b in zip(u.reshape(cols, rows, -1).split(max(1, cols // 64)), x.split(max(1, cols // 64))):
            g += torch.movedim(a, 1, 0).reshape(rows, -1) @ b.reshape(-1, nd.r)
        om[nd.v] = drm.Yt(nd.v).T @ g
        ps[nd.v] = g if nd.leaf else _psi(lay, drm, nd, g, [nd.r])
    ps[0] = _psi(lay, drm, lay.nodes[0], t, [])
    return om, ps


def _sketch_cp(lay, drm, w, a):
    """(Omega, Psi) of sum_q w_q a_1q o ... o a_dq."""
    x = [f.T @ m for f, m in zip(drm.X, a)]
    y = [f.T @ m for f, m in zip(drm.Y, a)]
    prod = lambda vs: torch.stack(vs).prod(0)
    yt = lambda nd: _kr([a[mu] for mu in range(nd.lo, nd.hi)]) if nd.identity else prod(y[nd.lo:nd.hi])[:nd.s]
    om, ps = {}, {}
    for nd in lay.nodes:
        if not nd.sketched and nd.parent >= 0:
            continue
        tail = [] if nd.parent < 0 else [prod(x[:nd.lo] + x[nd.hi:])[:nd.r]]
        head = [_kr([a[mu] for mu in range(nd.lo, nd.hi)])] if nd.leaf else [yt(lay.nodes[c]) for c in nd.ch]
        ps[nd.v] = (_kr(head + tail) @ w).reshape(lay.psi_shape(nd))
        if nd.sketched:
            om[nd.v] = (yt(nd) * w) @ tail[0].T
    return om, ps


def _sketch_ttn(lay, drm, cores):
    """(Omega, Psi) of a tensor in tree format, by an up and a down sweep over its cores."""
    nodes, ux, uy, env, om, ps = lay.nodes, {}, {}, {}, {}, {}

    def against(core, mats, axis):
        """The core with the axes from `axis` on contracted, all against the same column index."""
        out = torch.tensordot(core, mats[-1], dims=([core.ndim - 1], [0]))
        for m in reversed(mats[:-1]):
            out = torch.einsum("...bj,bj->...j", out, m)
        return out

    for nd in sorted(nodes, key=lambda n: -n.v):
        if nd.parent < 0:
            continue
        if nd.leaf:
            ux[nd.v] = cores[nd.v] @ _kr(drm.X[nd.lo:nd.hi])
            uy[nd.v] = cores[nd.v] @ _kr(drm.Y[nd.lo:nd.hi])
        else:
            ux[nd.v] = against(cores[nd.v], [ux[c] for c in nd.ch], 1)
            uy[nd.v] = against(cores[nd.v], [uy[c] for c in nd.ch], 1)
    for nd in nodes:                                        # parents come before their children
        for k, c in enumerate(nd.ch):
            core, mats = cores[nd.v], [ux[o] for o in nd.ch if o != c]
            if nd.parent >= 0:
                core, mats, k = core, [env[nd.v]] + mats, k + 1
            env[c] = against(torch.movedim(core, k, 0), mats, 1)
    for nd in nodes:
        if not nd.sketched and nd.parent >= 0:
            continue
        if nd.sketched:
            e = env[nd.v][:, :nd.r]
            om[nd.v] = uy[nd.v][:, :nd.s].T @ e
            p = torch.tensordot(cores[nd.v], e, dims=([0], [0]))
        else:
            p = cores[nd.v]
        for k, c in enumerate(nd.ch):
            p = _on_axis(p, k, cores[c] if nodes[c].identity else uy[c][:, :nodes[c].s])
        ps[nd.v] = p
    return om, ps


def _flat(lay, om, ps):
    """The state buffer's order: per node in level order Omega then Psi (the root: Psi)."""
    return torch.cat([x for v in lay.order if v in ps for x in (([om[v].reshape(-1)] if v in om else []) + [ps[v].reshape(-1)])])


def _cores(lay, om, ps):
    """Cores from the sketches: QR with diag(R) >= 0, pseudo-inverse above 10 u ||R||, assembly."""
    q, rp = {}, {}
    for nd in lay.nodes:
        if nd.sketched:
            a, b = torch.linalg.qr(om[nd.v])
            sign = torch.where(torch.diagonal(b) < 0, -1.0, 1.0).double()
            q[nd.v], b = a * sign, b * sign[:, None]
            u, s, vt = torch.linalg.svd(b)
            keep = s > 10 * 2.0 ** -52 * s[0]
            rp[nd.v] = (vt[keep].T / s[keep]) @ u[:, keep].T
    out = []
    for v in lay.order:
        nd = lay.nodes[v]
        if nd.identity:
            out.append(torch.eye(nd.n, dtype=torch.float64, device="cuda"))
            continue
        p = ps[v]
        for k, c in enumerate(nd.ch):
            if not lay.nodes[c].identity:
                p = _on_axis(p, k, q[c])
        out.append(torch.movedim(_on_axis(p, p.ndim - 1, rp[v]), -1, 0) if nd.parent >= 0 else p)
    return torch.cat([x.reshape(-1) for x in out])


def _unflat(lay, acc):
    om, ps, at = {}, {}, 0
    for v in lay.order:
        nd = lay.nodes[v]
        if nd.sketched:
            om[v] = acc[at:at + nd.s * nd.r].reshape(nd.s, nd.r)
            at += nd.s * nd.r
        if nd.sketched or nd.parent < 0:
            shape = lay.psi_shape(nd)
            ps[v] = acc[at:at + math.prod(shape)].reshape(shape)
            at += math.prod(shape)
    return om, ps


def _box_sketch(lay, seed, fmt, data, off, ext):
    """The sketch of a box: the rows of the box in every factor and block; leaf and identity axes put in their place."""
    om, ps = _sketch_dense(lay, _Drm(lay, seed, fmt, True, off, ext), data)
    for nd in lay.nodes:
        if nd.v in ps and nd.leaf:
            box = torch.zeros(lay.dims[nd.lo:nd.hi] + [nd.r], dtype=torch.float64, device="cuda")
            box[tuple(slice(off[mu], off[mu] + ext[mu]) for mu in range(nd.lo, nd.hi))] = ps[nd.v].reshape([ext[mu] for mu in range(nd.lo, nd.hi)] + [nd.r])
            ps[nd.v] = box.reshape(nd.n, nd.r)
    return _flat(lay, om, ps)


def _dequantised(x, lay):
    """What an E4M3 plan sketches: per 128 x 128 tile s = max / 448 and q = e4m3(x / s) in binary32, then bf16(q s)."""
    rows = math.prod(lay.dims[:lay.left.stop])
    m = x.reshape(rows, -1)
    cols = m.shape[1]
    m = torch.nn.functional.pad(m, (0, -cols % 128, 0, -rows % 128)).reshape(-(-rows // 128), 128, -(-cols // 128), 128)
    top = m.abs().amax(dim=(1, 3), keepdim=True)
    s = torch.where(top > 0, top / torch.full_like(top, 448.0), torch.ones_like(top))    # a division, not a product with 1 / 448
    q = (m / s).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).float()
    return (q * s).to(torch.bfloat16).double().reshape(m.shape[0] * 128, -1)[:rows, :cols].reshape(lay.dims)


def exact(case, seed):
    fmt, drm_seed = case["fmt"], 2024 + seed
    if case["kind"] == "serve":
        mix = _mix(case)
        out = [0.0] * len(mix)
        for k, off, ext, data in _slices(case, mix, seed):
            out[k] = out[k] + _box_sketch(mix[k][0], drm_seed + k, "bf16", data.double(), off, ext)
        return out
    lay = _layout(case)
    if case["kind"] == "stream":
        out = 0.0
        drm = _Drm(lay, drm_seed, DRM[fmt], False)
        one = torch.ones(case["cp"], dtype=torch.float64, device="cuda")
        for cp, off, ext, box in _stream_updates(case, lay, seed):
            out = out + _flat(lay, *_sketch_cp(lay, drm, one, cp)) + _box_sketch(lay, drm_seed, DRM[fmt], box.double(), off, ext)
        return out
    if case["kind"] == "ttn":
        return _flat(lay, *_sketch_ttn(lay, _Drm(lay, drm_seed, DRM[fmt], False), _ttn_cores(lay, case["rank"], seed)))
    if case["kind"] == "recover":
        w, a = _cp_decaying(lay, case["decay"], seed)
        acc = _flat(lay, *_sketch_cp(lay, _Drm(lay, drm_seed, DRM[fmt], False), w, a))
        om, ps = _unflat(lay, acc if fmt == "f64" else acc.float().double())
        return _cores(lay, om, ps)
    data, off, ext = _box_tensor(case, lay, seed)
    if case["kind"] == "slab":
        return _box_sketch(lay, drm_seed, DRM[fmt], data.double(), off, ext)
    if fmt == "e4m3":
        t = _dequantised(data, lay)
    elif fmt == "bf16x2":
        hi = data.to(torch.bfloat16)
        t = hi.double() + (data - hi.float()).to(torch.bfloat16).double()
    else:
        t = data.double()
    del data
    om, ps = _sketch_dense(lay, _Drm(lay, drm_seed, DRM[fmt]), t)
    if fmt == "e4m3":
        return {"q": None, "scale": None, "state": _flat(lay, om, ps)}
    if case["kind"] == "whole":
        return {"state": _flat(lay, om, ps), "cores": _cores(lay, om, ps)}
    return _flat(lay, om, ps)

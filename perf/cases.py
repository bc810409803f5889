"""The calls whose speed is followed, with their inputs, results and bounds.

Each case is one call a user of the library makes: an axis permute, a reorder
or scatter by an index sequence, an interlace or de-interlace, a captured batch
of many small operations, or a stencil sweep.  listed() names the fixed ones,
draw() gives others of the same ranges.  Payloads are random bit patterns of
integer type (every operation but the stencil moves opaque elements), index
sequences are permutations, and stencil grids are standard-normal floats.
"""
import math

import torch

import paper_1011_3583_gb300 as rr

MIB = 1 << 20
_INT = {1: torch.uint8, 2: torch.int16, 4: torch.int32, 8: torch.int64}


def listed():
    return [
        # One matrix of 4 MB turned over, as between two layers of a solver:
        # the smallest call, where launch latency counts.
        dict(name="transpose_1024_fp32", kind="permute", elem=4, dims="1024,1024", perm="1,0"),
        # A rank-3 field with its axes rotated, the solver's or FFT's layout
        # change between sweeps, at the largest ordinary size.
        dict(name="permute_512cube_fp32", kind="permute", elem=4, dims="512,512,512", perm="1,2,0"),
        # A rank-4 half-precision tensor fully reversed: short planes, far
        # strides on both sides.
        dict(name="permute_64x128x256x64_2b", kind="permute", elem=2, dims="64,128,256,64", perm="3,2,1,0"),
        # A batch of three-channel byte images from planar (NCHW) to pixel
        # order (NHWC), the everyday conversion around a decoder or a network.
        dict(name="images_nchw_to_nhwc_u8", kind="permute", elem=1, dims="32,3,1024,1024", perm="0,2,3,1"),
        # Extents that are no multiple of anything, which leave ragged tiles
        # and unaligned rows.
        dict(name="permute_ragged_fp32", kind="permute", elem=4, dims="251,333,517", perm="2,0,1"),
        # Records put in sorted order by a permutation too large for any cache
        # (the tail end of a sort, a mesh renumbering).
        dict(name="reorder_2p28_fp32_random", kind="reorder", elem=4, n=1 << 28, pattern="random", idx_bytes=4),
        # A mesh renumbering of ordinary size whose source fits the L2.
        dict(name="reorder_3M_8b_random", kind="reorder", elem=8, n=3000017, pattern="random", idx_bytes=4),
        # The inverse direction: results written back to where they belong.
        dict(name="scatter_100M_fp32_random", kind="scatter", elem=4, n=100000007, pattern="random", idx_bytes=4),
        # Three byte planes of a picture joined into pixels.
        dict(name="interlace_4096sq_u8_k3", kind="interlace", elem=1, k=3, n=4096 * 4096),
        # Records of four floats split into arrays (AoS to SoA).
        dict(name="deinterlace_2p26_fp32_k4", kind="deinterlace", elem=4, k=4, n=1 << 26),
        # Thousands of small operations of uneven shapes replayed as one
        # captured batch, as a server or a data pipeline issues them.
        dict(name="batch_mix_2048", kind="batch", ops=2048, mix_seed=1),
        # One sweep of the finite-difference Laplacian of order II.
        dict(name="stencil_4096sq_order2", kind="stencil", ny=4096, nx=4096, taps="cross2", boundary="zero"),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _draw_shape(rng, rank, lo_total, hi_total, hi_extent):
    while True:
        dims = [_log_int(rng, 2, hi_extent) for _ in range(rank)]
        if rng.random() < 0.4:
            dims = [max(4, d // 16 * 16) for d in dims]
        if lo_total <= math.prod(dims) <= hi_total:
            return dims


def draw(rng):
    kind = rng.choice(["permute", "permute", "images", "reorder", "scatter", "interlace", "deinterlace", "batch",
                       "stencil"])
    if kind == "permute":
        elem = rng.choice([1, 2, 4, 8])
        rank = rng.choice([2, 3, 3, 4, 4, 5])
        total = _log_int(rng, MIB, 512 * MIB) // elem
        dims = _draw_shape(rng, rank, total // 2, total, 16384)
        while True:
            perm = list(range(rank))
            rng.shuffle(perm)
            if perm != sorted(perm):
                break
        return dict(kind="permute", elem=elem, dims=",".join(map(str, dims)), perm=",".join(map(str, perm)))
    if kind == "images":
        elem, c = rng.choice([1, 1, 2, 4]), rng.choice([1, 2, 3, 3, 4])
        h = _log_int(rng, 64, 1080)
        w = _log_int(rng, 64, 1920)
        if rng.random() < 0.7:
            w = w // 16 * 16
        n = max(1, min(256, _log_int(rng, MIB, 512 * MIB) // (h * w * c * elem)))
        if rng.random() < 0.5:
            return dict(kind="permute", elem=elem, dims=f"{n},{c},{h},{w}", perm="0,2,3,1")
        return dict(kind="permute", elem=elem, dims=f"{n},{h},{w},{c}", perm="0,3,1,2")
    if kind in ("reorder", "scatter"):
        elem = rng.choice([1, 2, 4, 4, 8, 16])
        cap = (512 if elem >= 4 else 64) * MIB // elem
        return dict(kind=kind, elem=elem, n=_log_int(rng, 65536, cap), pattern=rng.choice(["random", "random", "blocks"]),
                    idx_bytes=rng.choice([4, 4, 8]))
    if kind in ("interlace", "deinterlace"):
        elem, k = rng.choice([1, 2, 4, 8]), rng.choice([2, 3, 4, 5, 6, 8])
        n = _log_int(rng, MIB, 512 * MIB) // (elem * k)
        if rng.random() < 0.6:
            n = n // 256 * 256 + 256
        return dict(kind=kind, elem=elem, k=k, n=n)
    if kind == "batch":
        return dict(kind="batch", ops=_log_int(rng, 32, 2048), mix_seed=rng.randrange(1 << 30))
    nx = _log_int(rng, 512, 8192)
    if rng.random() < 0.7:
        nx = nx // 32 * 32
    return dict(kind="stencil", ny=_log_int(rng, 512, 8192), nx=nx,
                taps=rng.choice(["cross1", "cross2", "cross3", "cross4", "box1", "box2", "list17"]),
                boundary=rng.choice(["zero", "clamp"]))


# ---------------------------------------------------------------------------
# Shapes of a batch: permutes of rank 2-5, reorders and interlaces with
# k in {2, 3, 4}, elements of 1 to 8 bytes, extents log-uniform in [1, 512],
# element totals in [2^8, 2^22].

def _batch_ops(case):
    import random
    rng = random.Random(case["mix_seed"])

    def shape(lo):
        while True:
            dims = [_log_int(rng, 1, 512) for _ in range(rng.randint(2, 5))]
            if lo <= math.prod(dims) <= 1 << 22:
                return dims

    ops = []
    for _ in range(case["ops"]):
        kind, elem = rng.choice(["permute", "reorder", "interlace"]), rng.choice([1, 2, 4, 8])
        if kind == "permute":
            dims = shape(256)
            perm = list(range(len(dims)))
            rng.shuffle(perm)
            ops.append(dict(kind=kind, elem=elem, dims=dims, perm=perm, n=math.prod(dims), k=1))
        elif kind == "reorder":
            ops.append(dict(kind=kind, elem=elem, n=math.prod(shape(256)), k=1))
        else:
            k = rng.randint(2, 4)
            n = max(1, math.prod(shape(256 * k)) // k)
            ops.append(dict(kind=rng.choice(["interlace", "deinterlace"]), elem=elem, n=n, k=k))
    return ops


def _batch_layout(ops):
    """Byte offsets in the payload slabs (every plane on a 256-byte boundary)
    and element offsets in the index slab, and the slabs' sizes."""
    at, idx_at, pos, ipos = [], [], 0, 0
    for op in ops:
        planes = op["k"] if op["kind"] in ("interlace", "deinterlace") else 1
        step = -(-op["n"] * op["elem"] // 256) * 256
        at.append([pos + j * step for j in range(planes)])
        pos += planes * step
        idx_at.append(ipos)
        if op["kind"] == "reorder":
            ipos += -(-op["n"] // 64) * 64
    return at, idx_at, pos, ipos


# ---------------------------------------------------------------------------
# Inputs, the same for prepare() and exact().

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _payload(count, elem, g):
    """count elements of random bits; a 16-byte element is a row of two words."""
    if elem == 16:
        return torch.randint(-2 ** 62, 2 ** 62, (count, 2), dtype=torch.int64, device="cuda", generator=g)
    lo, hi = (0, 256) if elem == 1 else (-2 ** (8 * elem - 2), 2 ** (8 * elem - 2))
    return torch.randint(lo, hi, (count,), dtype=_INT[elem], device="cuda", generator=g)


def _permutation(case, g):
    n, dtype = case["n"], torch.int32 if case["idx_bytes"] == 4 else torch.int64
    if case["pattern"] == "blocks":  # runs of 4096 consecutive indices in random order, a shorter run last
        nb = n // 4096
        head = (torch.randperm(nb, device="cuda", generator=g)[:, None] * 4096
                + torch.arange(4096, device="cuda")[None, :]).reshape(-1)
        return torch.cat([head, torch.arange(nb * 4096, n, device="cuda")]).to(dtype)
    return torch.randperm(n, dtype=dtype, device="cuda", generator=g)


def _ints(text):
    return [int(x) for x in text.split(",")]


def _taps(name, seed):
    size = int("".join(ch for ch in name if ch.isdigit()))
    if name.startswith("box"):
        w = 1.0 / (2 * size + 1) ** 2
        return [(y, x, w) for y in range(-size, size + 1) for x in range(-size, size + 1)]
    if name.startswith("list"):  # scattered taps of a learned or measured filter
        g = torch.Generator().manual_seed(seed)
        at = torch.randperm(81, generator=g)[:size].tolist()
        w = torch.randn(size, generator=g).tolist()
        return [(p // 9 - 4, p % 9 - 4, v) for p, v in zip(at, w)]
    # central second differences of accuracy 2 * size, along both axes
    c = {1: [-2.0, 1.0], 2: [-5 / 2, 4 / 3, -1 / 12], 3: [-49 / 18, 3 / 2, -3 / 20, 1 / 90],
         4: [-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560]}[size]
    taps = [(0, 0, 2 * c[0])]
    for d in range(1, size + 1):
        taps += [(d, 0, c[d]), (-d, 0, c[d]), (0, d, c[d]), (0, -d, c[d])]
    return taps


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind == "permute":
        dims, perm = _ints(case["dims"]), _ints(case["perm"])
        src = _payload(math.prod(dims), case["elem"], g).view(dims)
        dst = torch.empty([dims[p] for p in perm], dtype=src.dtype, device="cuda")
        return dict(kind=kind, elem=case["elem"], dims=dims, perm=perm, src=src, dst=dst)
    if kind in ("reorder", "scatter"):
        src = _payload(case["n"], case["elem"], g)
        idx = _permutation(case, g)
        call = {("reorder", 4): rr.reorder, ("reorder", 8): rr.reorder64,
                ("scatter", 4): rr.scatter, ("scatter", 8): rr.scatter64}[kind, case["idx_bytes"]]
        return dict(kind=kind, elem=case["elem"], n=case["n"], src=src, idx=idx, dst=torch.zeros_like(src), call=call)
    if kind in ("interlace", "deinterlace"):
        n, k = case["n"], case["k"]
        planes = [_payload(n, case["elem"], g) for _ in range(k)] if kind == "interlace" else \
                 [torch.empty(n, dtype=_INT[case["elem"]], device="cuda") for _ in range(k)]
        joined = _payload(n * k, case["elem"], g) if kind == "deinterlace" else \
            torch.empty(n * k, dtype=_INT[case["elem"]], device="cuda")
        return dict(kind=kind, elem=case["elem"], n=n, planes=planes, joined=joined)
    if kind == "batch":
        src, idx, ops, (at, idx_at, nbytes, _) = _batch_inputs(case, g)
        dst = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        plan = rr.Plan()
        s, d, ix = src.data_ptr(), dst.data_ptr(), idx.data_ptr()
        for op, offs, io in zip(ops, at, idx_at):
            ins, outs = [s + o for o in offs], [d + o for o in offs]
            if op["kind"] == "permute":
                plan.add_permute(outs[0], ins[0], op["elem"], op["dims"], op["perm"])
            elif op["kind"] == "reorder":
                plan.add_reorder(outs[0], ins[0], ix + 4 * io, op["n"], op["elem"])
            elif op["kind"] == "interlace":
                plan.add_interlace(outs[0], ins, op["n"], op["elem"])
            else:
                plan.add_deinterlace(outs, ins[0], op["n"], op["elem"])
        plan.finalize(torch.cuda.current_stream().cuda_stream)
        return dict(kind=kind, plan=plan, src=src, idx=idx, dst=dst)
    src = torch.randn((case["ny"], case["nx"]), device="cuda", generator=g)
    return dict(kind=kind, src=src, dst=torch.empty_like(src), taps=_taps(case["taps"], seed),
                boundary=rr.STENCIL_CLAMP if case["boundary"] == "clamp" else rr.STENCIL_ZERO)


def _batch_inputs(case, g):
    ops = _batch_ops(case)
    layout = _batch_layout(ops)
    at, idx_at, nbytes, n_idx = layout
    src = torch.randint(-2 ** 62, 2 ** 62, (-(-nbytes // 8),), dtype=torch.int64, device="cuda", generator=g)
    idx = torch.zeros(max(1, n_idx), dtype=torch.int32, device="cuda")
    for op, io in zip(ops, idx_at):
        if op["kind"] == "reorder":
            torch.randperm(op["n"], generator=g, out=idx[io:io + op["n"]], dtype=torch.int32, device="cuda")
    return src.view(torch.uint8)[:nbytes], idx, ops, layout


def run(state):
    kind, stream = state["kind"], torch.cuda.current_stream().cuda_stream
    if kind == "permute":
        rr.permute(state["dst"], state["src"], state["elem"], state["dims"], state["perm"], stream)
        return state["dst"]
    if kind in ("reorder", "scatter"):
        state["call"](state["dst"], state["src"], state["idx"], state["n"], state["elem"], stream)
        return state["dst"]
    if kind == "interlace":
        rr.interlace(state["joined"], state["planes"], state["n"], state["elem"], stream)
        return state["joined"]
    if kind == "deinterlace":
        rr.deinterlace(state["planes"], state["joined"], state["n"], state["elem"], stream)
        return state["planes"]
    if kind == "batch":
        state["plan"].run(stream)
        return state["dst"]
    ny, nx = state["src"].shape
    rr.stencil2d(state["dst"], state["src"], ny, nx, state["taps"], state["boundary"], stream)
    return state["dst"]


def work(case):
    kind = case["kind"]
    if kind == "permute":
        return dict(bytes=2 * case["elem"] * math.prod(_ints(case["dims"])), flops=0)
    if kind in ("reorder", "scatter"):
        return dict(bytes=case["n"] * (2 * case["elem"] + case["idx_bytes"]), flops=0)
    if kind in ("interlace", "deinterlace"):
        return dict(bytes=2 * case["n"] * case["k"] * case["elem"], flops=0)
    if kind == "batch":
        return dict(bytes=sum(2 * op["n"] * op["k"] * op["elem"] + (4 * op["n"] if op["kind"] == "reorder" else 0)
                              for op in _batch_ops(case)), flops=0)
    cells = case["ny"] * case["nx"]
    return dict(bytes=8 * cells, flops=2 * len(_taps(case["taps"], 0)) * cells)


def tolerance(case):
    # The rearrangements move bits: every byte is the same.  A stencil sums at
    # most 25 products in fp32, in an order of its own: 6e-8 from 64-bit sums
    # on the listed grid.
    return {"rel": 3e-7, "max": 3e-6} if case["kind"] == "stencil" else "exact"


def exact(case, seed):
    """The results in plain torch (64-bit sums for the stencil)."""
    kind, g = case["kind"], _gen(seed)
    if kind == "permute":
        dims = _ints(case["dims"])
        return _payload(math.prod(dims), case["elem"], g).view(dims).permute(_ints(case["perm"])).contiguous()
    if kind in ("reorder", "scatter"):
        src = _payload(case["n"], case["elem"], g)
        idx = _permutation(case, g).long()
        if kind == "reorder":
            return src[idx]
        dst = torch.zeros_like(src)
        dst[idx] = src
        return dst
    if kind == "interlace":
        return torch.stack([_payload(case["n"], case["elem"], g) for _ in range(case["k"])], 1).reshape(-1)
    if kind == "deinterlace":
        joined = _payload(case["n"] * case["k"], case["elem"], g).view(case["n"], case["k"])
        return [joined[:, j].contiguous() for j in range(case["k"])]
    if kind == "batch":
        src, idx, ops, (at, idx_at, nbytes, _) = _batch_inputs(case, g)
        dst = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        for op, offs, io in zip(ops, at, idx_at):
            n, k, dt = op["n"], op["k"], _INT[op["elem"]]
            size = n * op["elem"]

            def part(slab, off, length):
                return slab[off:off + length].view(dt)

            if op["kind"] == "permute":
                part(dst, offs[0], size).copy_(
                    part(src, offs[0], size).view(op["dims"]).permute(op["perm"]).reshape(-1))
            elif op["kind"] == "reorder":
                part(dst, offs[0], size).copy_(part(src, offs[0], size)[idx[io:io + n].long()])
            elif op["kind"] == "interlace":
                part(dst, offs[0], size * k).copy_(torch.stack([part(src, o, size) for o in offs], 1).reshape(-1))
            else:
                joined = part(src, offs[0], size * k).view(n, k)
                for j, o in enumerate(offs):
                    part(dst, o, size).copy_(joined[:, j])
        return dst
    src = torch.randn((case["ny"], case["nx"]), device="cuda", generator=g).double()
    taps = _taps(case["taps"], seed)
    r = max(max(abs(dy), abs(dx)) for dy, dx, _ in taps)
    mode = "replicate" if case["boundary"] == "clamp" else "constant"
    pad = torch.nn.functional.pad(src[None, None], (r, r, r, r), mode=mode)[0, 0]
    out = torch.zeros_like(src)
    for dy, dx, w in taps:  # weights as the call takes them, in fp32
        w32 = torch.tensor(w, dtype=torch.float32).item()
        out += w32 * pad[r + dy:r + dy + case["ny"], r + dx:r + dx + case["nx"]]
    return out

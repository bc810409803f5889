"""Permutes off the 16-byte grid and of thin planes (span copies, interlaces of
a few planes) on the GPU, byte for byte against the oracle, at the sizes where
their units, words and lanes come out uneven."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import DevBuf, sync, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1011_3583_gb300 import build, librearr
    build.build()
    librearr.load()
    return librearr


@pytest.fixture(scope="module")
def orc():
    return oracle.get()


def check(lr, orc, e, dims, perm, src_off=0, dst_off=0):
    n = int(np.prod(dims))
    src = synth.random_elements(n % 1009, n, e)
    s, d = to_dev(src, src_off), DevBuf(n * e, dst_off, fill=0x55)
    lr.permute(d.ptr, s.ptr, e, dims, perm)
    sync()
    assert np.array_equal(d.download(), orc.permute(src, e, dims, perm)), (e, dims, perm, src_off, dst_off)


# odd planes; a rank-5 op with short axes on both sides; thin planes both ways;
# one unit with a single cell left over; output spans over several axes; a
# unit's whole axes on both sides (no ranges)
SPANS = [([257, 255], [1, 0]), ([1031, 1027], [1, 0]), ([61, 67, 129], [2, 0, 1]), ([5, 33, 7, 11, 63], [4, 1, 2, 0, 3]),
         ([3, 5, 129, 517], [0, 2, 3, 1]), ([3, 129, 517, 5], [0, 3, 1, 2]), ([9973, 9, 7], [0, 2, 1]),
         ([64 * 5 + 1, 64 * 7 + 1], [1, 0]), ([41, 23, 2, 4, 93], [1, 3, 0, 4, 2]), ([8193, 65], [1, 0]),
         ([31, 6, 16, 42, 4], [3, 4, 0, 1, 2]), ([7, 11, 13, 17, 19, 2], [5, 3, 1, 0, 2, 4])]


@pytest.mark.parametrize("e", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("dims,perm", SPANS)
def test_spans(lr, orc, e, dims, perm):
    check(lr, orc, e, dims, perm)


@pytest.mark.parametrize("e,src_off,dst_off", [(1, 1, 0), (1, 0, 3), (1, 7, 13), (2, 2, 6), (2, 14, 0), (4, 4, 8),
                                               (4, 12, 0), (8, 8, 8)])
def test_spans_unaligned(lr, orc, e, src_off, dst_off):
    """Base addresses off the grid: planes that would otherwise be 16-byte tiles."""
    for dims, perm in (([512, 1024], [1, 0]), ([64, 96, 320], [2, 1, 0]), ([4, 3, 64, 1024], [0, 2, 3, 1])):
        check(lr, orc, e, dims, perm, src_off, dst_off)


# Calls large enough (10 MB and more) to be cut into units of the full 16 KB:
# odd planes, an odd rank-3 rotation, thin planes, a base off the grid.
@pytest.mark.parametrize("e,dims,perm,src_off,dst_off", [
    (1, [3331, 4099], [1, 0], 0, 0), (1, [251, 133, 517], [2, 0, 1], 3, 5), (1, [262147, 9, 7], [0, 2, 1], 1, 0),
    (2, [2053, 4099], [1, 0], 0, 0), (2, [131, 233, 257], [2, 0, 1], 6, 2), (2, [131101, 11, 6], [0, 2, 1], 2, 4),
    (4, [2053, 2051], [1, 0], 0, 0), (4, [131, 133, 257], [2, 0, 1], 4, 8), (4, [65543, 13, 5], [0, 2, 1], 12, 0),
    (8, [1031, 2053], [1, 0], 8, 0)])
def test_full_units(lr, orc, e, dims, perm, src_off, dst_off):
    assert int(np.prod(dims)) * e > 608 * 16384
    check(lr, orc, e, dims, perm, src_off, dst_off)


# planes of few groups (576 cells, the fewest) and of one past a unit, two batch
# axes, k of every staging form
@pytest.mark.parametrize("e", [1, 2, 4, 8])
@pytest.mark.parametrize("k", [2, 3, 5, 6, 8])
def test_planes(lr, orc, e, k):
    for batch, p in (([37], 16448 // e), ([1201], 1024 // e), ([301], 576), ([301], 1024), ([3, 5], 65552 // e)):
        if len(batch) == 1:
            check(lr, orc, e, batch + [k, p], [0, 2, 1])
            check(lr, orc, e, batch + [p, k], [0, 2, 1])
        else:  # the batch axes change places, so they stay two
            check(lr, orc, e, [batch[0], batch[1], k, p], [1, 0, 3, 2])
            check(lr, orc, e, [batch[0], batch[1], p, k], [1, 0, 3, 2])


def test_boxes(lr, orc):
    """Sub-boxes: rows that are not dense in the input."""
    g = synth.rng(7)
    for e in (1, 2, 4):
        dims = [37, 190, 211]
        src = synth.random_elements(e, int(np.prod(dims)), e)
        s = to_dev(src)
        for order in ([2, 1, 0], [2, 0, 1], [1, 2, 0]):
            base = [int(g.integers(0, 5)) for _ in dims]
            rng = [d - b - int(g.integers(0, 9)) for d, b in zip(dims, base)]
            d = DevBuf(int(np.prod([rng[a] for a in order])) * e, 0, fill=0x55)
            lr.reorder_nm(d.ptr, s.ptr, e, dims, order, base, rng)
            sync()
            assert np.array_equal(d.download(), orc.reorder_nm(src, e, dims, order, base, rng)), (e, order, base, rng)


def test_capture(lr, orc):
    """A span copy and planes captured in a graph and replayed on new contents."""
    import torch
    cases = [(1, [61, 67, 129], [2, 0, 1]), (2, [64, 3, 4096], [0, 2, 1])]
    bufs = []
    for e, dims, perm in cases:
        n = int(np.prod(dims))
        bufs.append((DevBuf(n * e, fill=0), DevBuf(n * e, fill=0)))
    st = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        for (e, dims, perm), (s, d) in zip(cases, bufs):
            lr.permute(d.ptr, s.ptr, e, dims, perm, torch.cuda.current_stream())
    for seed in (1, 2):
        srcs = [synth.random_elements(seed, int(np.prod(dims)), e) for e, dims, _ in cases]
        for a, (s, _) in zip(srcs, bufs):
            s.upload(a)
        graph.replay()
        sync()
        for a, (e, dims, perm), (_, d) in zip(srcs, cases, bufs):
            assert np.array_equal(d.download(), orc.permute(a, e, dims, perm)), (seed, e, dims, perm)


def test_large_batch(lr, orc):
    """A plan large enough to be split over the batch's kernels: every op as its
    single call would compute it, replayed on new contents."""
    plan = lr.Plan()
    ops = []
    for i in range(20):  # 2048 units each
        e, n = (1, 2, 1, 4)[i % 4], (1 << 22) - i
        ops.append(dict(kind="scatter" if i % 5 == 4 else "reorder", e=e, n=n, idx=synth.random_permutation(i, n)))
    for i in range(60):
        dims, perm = SPANS[i % len(SPANS)]
        ops.append(dict(kind="permute", e=(1, 2, 4, 8)[i % 4], n=int(np.prod(dims)), dims=dims, perm=perm))
    for dims, perm in (([64, 64, 128], [2, 1, 0]), ([128, 40, 256], [1, 0, 2]), ([70000], [0])):
        ops.append(dict(kind="permute", e=4, n=int(np.prod(dims)), dims=dims, perm=perm))
    for k in (2, 3, 9):
        ops.append(dict(kind="interlace", e=2, n=20000 + k, k=k))
    for op in ops:
        e, n = op["e"], op["n"]
        op["in"] = [DevBuf(n * e) for _ in range(op.get("k", 1))]
        op["out"] = DevBuf(n * e * op.get("k", 1), fill=0x55)
        if op["kind"] in ("reorder", "scatter"):
            op["didx"] = to_dev(op["idx"])
            add = plan.add_reorder if op["kind"] == "reorder" else plan.add_scatter
            add(op["out"].ptr, op["in"][0].ptr, op["didx"].ptr, n, e)
        elif op["kind"] == "permute":
            plan.add_permute(op["out"].ptr, op["in"][0].ptr, e, op["dims"], op["perm"])
        else:
            plan.add_interlace(op["out"].ptr, [b.ptr for b in op["in"]], n, e)
    assert plan.stats()[1] > 40000
    plan.finalize()
    for replay in range(2):
        for i, op in enumerate(ops):
            op["src"] = [synth.random_elements(1000 * replay + i + 7 * j, op["n"], op["e"]) for j in range(len(op["in"]))]
            for b, a in zip(op["in"], op["src"]):
                b.upload(a)
        before = lr.launch_count()
        plan.run()
        assert lr.launch_count() - before == 3  # split: gathers, the rest, span copies
        sync()
        for op in ops:
            e, n, src = op["e"], op["n"], op["src"]
            if op["kind"] == "reorder":
                want = orc.reorder(src[0], op["idx"], e)
            elif op["kind"] == "scatter":
                inv = np.empty(n, dtype=np.uint32)
                inv[op["idx"]] = np.arange(n, dtype=np.uint32)
                want = orc.reorder(src[0], inv, e)
            elif op["kind"] == "permute":
                want = orc.permute(src[0], e, op["dims"], op["perm"])
            else:
                want = orc.interlace(src, n, e)
            assert np.array_equal(op["out"].download(), want), (replay, op["kind"], e, n, op.get("dims"))


@pytest.mark.parametrize("others,kernels", [(0, 1), (3, 2)])
def test_split_without_spans(lr, orc, others, kernels):
    """Plans that are split but leave a kernel without ops: index gathers alone,
    and with interlaces and full tiles beside them."""
    plan = lr.Plan()
    want = []
    for i in range(21):  # 2048 units each
        n = (1 << 22) - i
        src, idx = synth.random_elements(i, n, 1), synth.random_permutation(i, n)
        d = DevBuf(n, fill=0x55)
        bufs = (to_dev(src), to_dev(idx), d)
        plan.add_reorder(d.ptr, bufs[0].ptr, bufs[1].ptr, n, 1)
        want.append((bufs, d, orc.reorder(src, idx, 1)))
    for i in range(others):
        dims, perm = ([128, 64, 256], [2, 0, 1]) if i % 2 else ([256, 512], [1, 0])
        n = int(np.prod(dims))
        src = synth.random_elements(50 + i, n, 4)
        s, d = to_dev(src), DevBuf(n * 4, fill=0x55)
        plan.add_permute(d.ptr, s.ptr, 4, dims, perm)
        want.append((s, d, orc.permute(src, 4, dims, perm)))
    plan.finalize()
    before = lr.launch_count()
    plan.run()
    assert lr.launch_count() - before == kernels
    sync()
    for _, d, w in want:
        assert np.array_equal(d.download(), w)

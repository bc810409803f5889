"""Large scatters (chunk lists) on the GPU: every written element must carry the
tag of a source whose index names it, every other element must be untouched."""
import numpy as np
import pytest

import synth
from tests.gpu_util import DevBuf, sync, to_dev

pytestmark = pytest.mark.gpu

MIN = 128 << 20  # bytes from which scatters leave the direct kernel


@pytest.fixture(scope="module")
def lr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1011_3583_gb300 import build, librearr
    build.build()
    librearr.load()
    return librearr


def check(lr, e, idx, dst_off=0):
    n, tag = idx.size, np.uint32 if e == 4 else np.uint64
    d = DevBuf(n * e, dst_off, fill=0xA7)
    s, ix = to_dev(np.arange(n, dtype=tag)), to_dev(idx)
    (lr.scatter64 if idx.dtype == np.uint64 else lr.scatter)(d.ptr, s.ptr, ix.ptr, n, e)
    sync()
    got = d.download().view(tag)
    hit = np.zeros(n, dtype=bool)
    hit[idx] = True
    assert np.all(got[~hit] == np.frombuffer(b"\xa7" * e, dtype=tag)[0])
    at = np.flatnonzero(hit)
    assert np.all(got[at] < n)
    assert np.array_equal(idx[got[at].astype(np.int64)].astype(np.int64), at)


# the smallest size, one element more (a tile and a chunk of little), a tile
# boundary, and one where the chunks are evened out to several rounds
@pytest.mark.parametrize("e,n", [(4, MIN // 4), (4, MIN // 4 + 1), (4, 24576 * 1400), (4, 50_000_017),
                                 (8, MIN // 8 + 3), (8, 16384 * 1100 - 1)])
@pytest.mark.parametrize("wide", [False, True])
def test_permutations(lr, e, n, wide):
    idx = synth.random_permutation(n % 97, n)
    check(lr, e, idx.astype(np.uint64) if wide else idx)


def test_unaligned_destination(lr):
    n = MIN // 4 + 4099
    for off in (4, 8, 12):
        check(lr, 4, synth.random_permutation(off, n), dst_off=off)


@pytest.mark.parametrize("e", [4, 8])
def test_repeats(lr, e):
    """Uniform repeats (lists part empty, part beyond a chunk's size), a range
    that the sample shows crowded, and one that only a list's overflow shows."""
    n = MIN // e + 12345
    check(lr, e, synth.random_indices(1, n, n))
    check(lr, e, synth.random_indices(2, n, n // 8) + np.uint32(n // 3))
    p = synth.random_permutation(3, n)
    lo = n // 2
    away = (p >= lo + 200_000) & (p < lo + 240_000)
    p[away] = lo + p[away] % np.uint32(40_000 // (e // 4))  # these chunks get more than their lists hold
    check(lr, e, p)
    p = synth.random_permutation(4, n)
    p[: n // 2] = np.uint32(77)
    check(lr, e, p)


@pytest.mark.parametrize("e", [4, 8])
def test_crowded(lr, e):
    """Repeats that crowd some chunks: all of them moderately (within the lists'
    room), a few far beyond it (stored past their lists), and so many that the
    bucketed passes run."""
    n = MIN // e + 4321
    g = synth.rng(e)
    check(lr, e, synth.random_indices(1, n, n * 3 // 4))
    p = synth.random_indices(2, n, n)
    hot = g.random(n) < 0.02
    p[hot] = n // 3 + p[hot] % np.uint32(3000)
    check(lr, e, p)
    p = synth.random_indices(3, n, n)
    w = np.uint32(n // 1000)
    hot = g.random(n) < 0.1
    p[hot] = p[hot] // w // np.uint32(40) * np.uint32(40) * w + p[hot] % w
    check(lr, e, p)
    check(lr, e, synth.random_indices(4, n, n // 3))
    check(lr, e, synth.random_indices(5, n, n // 2).astype(np.uint64))


@pytest.mark.parametrize("e", [4, 8])
@pytest.mark.parametrize("step", [17, 31, 1001])
def test_strides(lr, e, step):
    """Orders of a fixed stride, where a warp's indices rank in one list."""
    n = MIN // e + 4097
    while np.gcd(step, n) != 1:
        step += 1
    check(lr, e, (np.arange(n, dtype=np.uint64) * np.uint64(step) % np.uint64(n)).astype(np.uint32))


@pytest.mark.parametrize("form", ["scatter", "reorder"])
def test_capture(lr, form):
    """The whole pass sequence captured in a graph and replayed on sequences that
    take each of its branches: random, local, crowded."""
    import torch
    n = MIN // 4 + 77
    s, ix, d = DevBuf(n * 4, fill=0), DevBuf(n * 4, fill=0), DevBuf(n * 4, fill=0)
    call = getattr(lr, form)
    call(d.ptr, s.ptr, ix.ptr, n, 4)  # set-up outside the capture
    sync()
    st = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        call(d.ptr, s.ptr, ix.ptr, n, 4, torch.cuda.current_stream())
    blocks = (synth.random_permutation(5, n // 4096)[:, None].astype(np.uint32) * np.uint32(4096)
              + np.arange(4096, dtype=np.uint32)).reshape(-1)
    local = np.concatenate([blocks, np.arange(blocks.size, n, dtype=np.uint32)])
    for seed, idx in enumerate((synth.random_permutation(6, n), local, synth.random_indices(7, n, n // 3),
                                synth.random_permutation(8, n))):
        src = synth.random_elements(seed, n, 4)
        s.upload(src)
        ix.upload(idx)
        graph.replay()
        sync()
        got, src = d.download().view(np.uint32), src.view(np.uint32)
        if form == "reorder":
            assert np.array_equal(got, src[idx]), seed
        elif np.unique(idx).size == n:
            assert np.array_equal(got[idx], src), seed
        else:  # each written element carries a source that names it (values are unique enough to look up)
            key = (idx.astype(np.uint64) << np.uint64(32)) | src
            key.sort()
            at = np.unique(idx)
            want = (at.astype(np.uint64) << np.uint64(32)) | got[at]
            pos = np.searchsorted(key, want)
            assert np.array_equal(key[np.minimum(pos, n - 1)], want), seed


def test_two_threads(lr):
    """Calls of different sizes (so of different shared-memory needs) from two
    threads at a time."""
    import threading

    import torch
    jobs = []
    for n in (MIN // 4 + 77, 50_000_017):
        idx = synth.random_permutation(n % 89, n)
        d, s, ix = DevBuf(n * 4, fill=0xA7), to_dev(np.arange(n, dtype=np.uint32)), to_dev(idx)
        jobs.append((n, idx, d, s, ix, torch.cuda.Stream()))
    sync()
    errors = []

    def work(n, idx, d, s, ix, st):
        try:
            for _ in range(50):
                lr.scatter(d.ptr, s.ptr, ix.ptr, n, 4, stream=st.cuda_stream)
        except Exception as ex:  # reported by the test's thread
            errors.append(ex)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    sync()
    assert not errors, errors
    for n, idx, d, s, ix, st in jobs:
        got = d.download().view(np.uint32)
        assert np.array_equal(idx[got], np.arange(n, dtype=np.uint32))

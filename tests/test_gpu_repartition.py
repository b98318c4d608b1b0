"""ja_repartition at every alignment (whole words, shifted words, row ends) and with its slabs in the kernel's parameters or in a
device table: bit-exact against the oracle's packing."""
import numpy as np
import pytest
import torch

import paper_2609_03905_b200 as ja
import synth_inputs as si
from oracle import blocked

from gpu_util import check_status, download_bits, empty_like_tiling, np_bits, upload

pytestmark = pytest.mark.gpu
ES = blocked.equal_splits
BF, F32, F16 = torch.bfloat16, torch.float32, torch.float16


@pytest.mark.parametrize("dtype", [BF, F32])
@pytest.mark.parametrize("ext,src,dst", [
    ([64, 1], [1, 1], [4, 1]), ([7, 3], [1, 1], [2, 3]), ([65, 129], [3, 2], [1, 5]), ([257, 1023], [4, 1], [1, 8]), ([300, 2049], [7, 3], [2, 1]),
    ([128, 256], [2, 4], [4, 1]), ([1000, 37], [1, 1], [100, 1]), ([999, 515], [128, 2], [64, 32]),          # the last: a device table
    ([5, 33, 17], [1, 2, 3], [5, 1, 2]), ([3, 4, 9, 11], [1, 2, 1, 3], [3, 1, 2, 1]), ([4096, 40], [1024, 1], [3, 1]),
])
@pytest.mark.parametrize("once", [False, True])
def test_any_alignment(ext, src, dst, dtype, once):
    def move(x, y):
        if once:
            ja.ja_repartition_once(x.handle, y.handle, torch.cuda.current_stream().cuda_stream)
        else:
            ja.repartition(x, y)
    s_sp, d_sp = [ES(e, g) for e, g in zip(ext, src)], [ES(e, g) for e, g in zip(ext, dst)]
    x = si.normal(tuple(ext), 0.0, 1.0, dtype, 37, 1)
    a, b, c = upload(x, s_sp), empty_like_tiling(ext, d_sp, dtype), empty_like_tiling(ext, s_sp, dtype)
    move(a, b)
    assert np.array_equal(download_bits(b), blocked.pack(np_bits(x), d_sp))
    move(b, c)
    assert np.array_equal(download_bits(c), blocked.pack(np_bits(x), s_sp))
    check_status()          # guard zones around every payload


@pytest.mark.parametrize("dtype", [BF, F32])
@pytest.mark.parametrize("n,cuts", [(200, 13), (200, 24), (900, 60)])   # more shapes of slabs than a launch holds; more slabs; more than a few launches hold
def test_many_shapes(n, cuts, dtype):
    rng = np.random.default_rng(5)
    s_sp, d_sp = ([[0] + sorted(rng.choice(np.arange(1, n), cuts - 1, replace=False).tolist()) + [n] for _ in range(2)] for _ in range(2))
    x = si.normal((n, n), 0.0, 1.0, dtype, 37, 5)
    a, b, c = upload(x, s_sp), empty_like_tiling([n, n], d_sp, dtype), empty_like_tiling([n, n], d_sp, dtype)
    for _ in range(2):
        ja.repartition(a, b)
    ja.ja_repartition_once(a.handle, c.handle, torch.cuda.current_stream().cuda_stream)
    want = blocked.pack(np_bits(x), d_sp)
    assert np.array_equal(download_bits(b), want) and np.array_equal(download_bits(c), want)
    check_status()


@pytest.mark.parametrize("shape,cuts,dtype", [((97, 41), (4, 3), BF), ((1024, 512), (8, 4), F16), ((333,), (5,), F32)])
def test_dense_round_trip(shape, cuts, dtype):
    x = si.normal(shape, 0.0, 1.0, dtype, 37, 2)
    rel = ja.from_dense(x.cuda(), [ES(e, g) for e, g in zip(shape, cuts)])
    assert np.array_equal(np_bits(rel.payload.cpu()), blocked.pack(np_bits(x), rel.splits))
    back = ja.to_dense(rel)
    assert back.shape == x.shape and back.is_contiguous() and torch.equal(back.cpu(), x)


def test_first_use_inside_a_capture_and_replay_after_the_plan_is_gone():
    x = si.normal((130, 70), 0.0, 1.0, BF, 37, 3)
    s_sp, d_sp = [ES(130, 2), ES(70, 1)], [ES(130, 1), ES(70, 4)]
    a, b = upload(x, s_sp), empty_like_tiling([130, 70], d_sp, BF)
    w1, w2 = upload(x, s_sp), empty_like_tiling([130, 70], d_sp, BF)
    ja.repartition(w1, w2)                                   # the kernel's module is loaded
    c = ja.Relation([130, 70], d_sp, BF, b.payload)          # another handle on the same payload
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ja.repartition(a, c)
    c.close()                                                # drops the cached plan, not the captured launch
    b.payload.zero_()
    g.replay()
    assert np.array_equal(download_bits(b), blocked.pack(np_bits(x), d_sp))
    check_status()


def test_every_call_of_a_pair_costs_the_same():
    """4096 slabs: the first call makes the table that every later one reads, captured or not (one launch each); relations that meet
    once make none (a launch per 960 slabs)."""
    ext, s_sp, d_sp = [999, 515], [ES(999, 128), ES(515, 2)], [ES(999, 64), ES(515, 32)]
    x = si.normal(tuple(ext), 0.0, 1.0, BF, 37, 4)
    a, b = upload(x, s_sp), empty_like_tiling(ext, d_sp, BF)

    def launches(call):
        before = ja.ja_launch_count()
        call()
        return ja.ja_launch_count() - before

    stream = torch.cuda.current_stream().cuda_stream
    assert launches(lambda: ja.ja_repartition_once(a.handle, b.handle, stream)) == 5
    assert [launches(lambda: ja.repartition(a, b)) for _ in range(3)] == [1, 1, 1]
    g = torch.cuda.CUDAGraph()
    c = empty_like_tiling(ext, d_sp, BF)
    ja.repartition(a, c)
    with torch.cuda.graph(g):                                  # after ONE call of the pair
        assert launches(lambda: ja.repartition(a, c)) == 1
    c.payload.zero_()
    g.replay()
    want = blocked.pack(np_bits(x), d_sp)
    assert np.array_equal(download_bits(b), want) and np.array_equal(download_bits(c), want)
    check_status()


def test_a_small_pair_on_several_streams_and_in_a_graph():
    """Few slabs: the second call copies a table that only its stream reads; other streams, captures and a second pair in the memory of a
    closed one carry the slabs in parameters or in tables of their own."""
    ext, s_sp, d_sp = [300, 260], [ES(300, 3), ES(260, 2)], [ES(300, 2), ES(260, 5)]
    want = None
    for trial in range(3):
        x = si.normal(tuple(ext), 0.0, 1.0, BF, 37, 6 + trial)
        a, b = upload(x, s_sp), empty_like_tiling(ext, d_sp, BF)
        want = blocked.pack(np_bits(x), d_sp)
        streams = [torch.cuda.Stream() for _ in range(3)]
        torch.cuda.synchronize()
        for st in [streams[0], streams[0], streams[1], streams[0], streams[2], streams[1]]:
            b.payload.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(st):
                ja.repartition(a, b)
            torch.cuda.synchronize()
            assert np.array_equal(download_bits(b), want)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[0]):
            ja.repartition(a, b)
        b.payload.zero_()
        g.replay()
        assert np.array_equal(download_bits(b), want)
        a.close(), b.close()
    check_status()

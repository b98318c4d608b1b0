"""Products of 16-bit relations that TMA cannot address as they lie, on copies that it can (k_stage.cu), and the stores that go with them, against
an fp64 product of the same 16-bit inputs. Tolerance: gpu_util.TOL, ten half-ulps of the stored type; f32 accumulation does not show
beside it."""
import time

import numpy as np
import pytest
import torch

import paper_2609_03905_b200 as ja
import synth_inputs as si
from oracle import blocked

from gpu_util import TOL, check_status, download, empty_like_tiling, relfro, upload

pytestmark = pytest.mark.gpu
ES = blocked.equal_splits
BF, F16 = torch.bfloat16, torch.float16


def _problem(ti, tj, tk, dtype):
    m, k, n = ti[-1], tj[-1], tk[-1]
    a, b = si.normal((m, k), 0.0, 1.0, dtype, 37, 40), si.normal((k, n), 0.0, 1.0, dtype, 37, 41)
    res = empty_like_tiling([m, n], [ti, tk], dtype, fill=float("nan"))
    return a, b, upload(a, [ti, tj]), upload(b, [tj, tk]), res, ja.Spec("ij,jk->ik", {"i": ti, "j": tj, "k": tk})


def _check(res, a, b, dtype):
    got, ref = download(res), si.to_f64(a) @ si.to_f64(b)
    check_status()
    assert relfro(got, ref) <= TOL[dtype]
    ulp = 2.0 ** (-7 if dtype == BF else -10)      # of the largest value: a misplaced cell is far outside it
    assert np.abs(got - ref).max() <= ulp * np.abs(ref).max()


# which operand is copied (odd columns of either or both, rows in unequal blocks), remainders of tiles, stages and 16-byte words, words that
# cross split points, blocks narrower than a word, one and two CTAs a tile, the last tiles split, few rows
@pytest.mark.parametrize("ti,tj,tk", [
    (ES(1000, 1), ES(2001, 1), ES(1504, 1)),                 # A alone has odd rows
    (ES(1000, 1), ES(2000, 1), ES(1501, 1)),                 # B alone
    (ES(1025, 1), ES(2001, 1), ES(1281, 1)),                 # both, one past a tile
    (ES(1500, 2), ES(2503, 2), ES(2001, 2)),                 # odd halves
    (ES(4001, 4), ES(3000, 1), ES(2504, 1)),                 # unequal row blocks only
    ([0, 100, 1301], [0, 130, 1931], [0, 135, 271, 1400]),   # ragged
    (ES(1640, 3), list(range(0, 1407, 7)), ES(1520, 2)),     # contracted intervals shorter than a 16-byte word
    (ES(1640, 3), ES(1699, 1), list(range(0, 1407, 7))),     # and columns
    (ES(1024, 1), ES(2200, 8), ES(1024, 4)),                 # contracted blocks of 275 rows in four columns of blocks: B is copied as well
    (ES(1024, 1), ES(2200, 8), ES(1024, 1)),                 # in one: B stays, as one block
    (ES(1280, 10), ES(4416, 4), ES(1511, 1)),                # A stays, B copied with A's contracted blocks
    (ES(4097, 7), ES(4416, 4), ES(3072, 4)),                 # B stays in its blocks, A copied with them
    (ES(4097, 1), ES(321, 1), ES(4351, 1)),                  # more tiles than pairs of SMs, and a short contracted index
    (ES(30, 1), ES(4001, 1), ES(3501, 1)),                   # few rows
    (ES(1, 1), ES(5001, 1), ES(3999, 3)),
    (ES(65, 5), ES(3999, 1), ES(3000, 5)),                   # few rows in several blocks
])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_copied_operands(ti, tj, tk, dtype):
    a, b, ra, rb, res, spec = _problem(ti, tj, tk, dtype)
    before = ja.ja_launch_count()
    spec.execute([ra, rb], res)
    assert ja.ja_launch_count() - before >= 2               # a copy and a product
    _check(res, a, b, dtype)


def test_captures():
    """A capture cannot take the scratch of the copies: before any other call it records the form without them, afterwards the copies."""
    a, b, ra, rb, res, first = _problem(ES(1000, 1), ES(2001, 1), ES(1501, 1), BF)
    first.execute([ra, rb], res)                 # puts the relations' key tables on the device, which a capture cannot either
    torch.cuda.current_stream().synchronize()
    spec = ja.Spec("ij,jk->ik", {"i": ES(1000, 1), "j": ES(2001, 1), "k": ES(1501, 1)}, "mul", (), "sum")
    st = torch.cuda.Stream()
    for launches in (1, 2):
        with torch.cuda.stream(st):
            g = torch.cuda.CUDAGraph()
            before = ja.ja_launch_count()
            with torch.cuda.graph(g, stream=st):
                spec.execute([ra, rb], res)
            assert ja.ja_launch_count() - before == launches
            res.payload.fill_(float("nan"))
            g.replay()
            st.synchronize()
            _check(res, a, b, BF)
            res.payload.fill_(float("nan"))
            spec.execute([ra, rb], res)
            st.synchronize()
            _check(res, a, b, BF)


def test_one_plan_on_two_streams_and_many_calls_in_a_row():
    """Scratch taken on one stream serves another one behind it, and a queue of calls of several plans gives each its own result."""
    sets = [_problem(ES(1300, 2), ES(1501, 1), ES(1401, 3), BF) for _ in range(2)]
    other = torch.cuda.Stream()
    for k in range(20):
        _, _, ra, rb, res, spec = sets[k % 2]
        spec.execute([ra, rb], res)
    torch.cuda.current_stream().synchronize()
    for a, b, ra, rb, res, spec in sets:
        _check(res, a, b, BF)
        res.payload.fill_(float("nan"))
        torch.cuda.current_stream().synchronize()
        with torch.cuda.stream(other):
            spec.execute([ra, rb], res)
            other.synchronize()
        _check(res, a, b, BF)


def test_streams_ordered_by_events_alone():
    """The second stream's call neither waits on the host for the first stream nor starts before it."""
    a, b, ra, rb, res, spec = _problem(ES(1300, 2), ES(1501, 1), ES(1401, 3), BF)
    a2, b2, ra2, rb2, res2, spec2 = _problem(ES(30, 1), ES(4001, 1), ES(3501, 1), BF)
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    for p in ((ra, rb, res, spec), (ra2, rb2, res2, spec2)):   # the key tables and the modules, which the host does wait for
        ja.Spec("ij,jk->ik", p[3].parts).execute([p[0], p[1]], p[2])
    torch.cuda.synchronize()
    payloads = {r: r.payload.clone() for r in (ra, rb)}
    for r in payloads:
        r.payload.fill_(float("nan"))
    res.payload.fill_(float("nan"))
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        torch.cuda._sleep(400_000_000)             # a fifth of a second
        spec2.execute([ra2, rb2], res2)
        spec.execute([ra, rb], res)                # of operands that are not there yet
        for r, x in payloads.items():
            r.payload.copy_(x)
        done = first.record_event()
    second.wait_event(done)
    with torch.cuda.stream(second):
        spec.execute([ra, rb], res)
        spec2.execute([ra2, rb2], res2)
    assert not done.query()                        # the host is here before the first stream is done
    second.synchronize()
    _check(res, a, b, BF)
    _check(res2, a2, b2, BF)


def test_first_stream_may_be_gone():
    from cuda.bindings import runtime as rt
    a, b, ra, rb, res, spec = _problem(ES(1300, 2), ES(1501, 1), ES(1401, 3), BF)
    err, gone = rt.cudaStreamCreateWithFlags(rt.cudaStreamNonBlocking)
    torch.cuda.synchronize()
    spec.execute([ra, rb], res, stream=int(gone))
    assert rt.cudaStreamSynchronize(gone)[0] == rt.cudaStreamDestroy(gone)[0] == err == rt.cudaError_t.cudaSuccess
    _check(res, a, b, BF)
    res.payload.fill_(float("nan"))
    before = ja.ja_launch_count()
    spec.execute([ra, rb], res)
    assert ja.ja_launch_count() - before == 2
    _check(res, a, b, BF)


def test_capture_on_another_stream_than_the_first_call():
    a, b, ra, rb, res, spec = _problem(ES(1000, 1), ES(2001, 1), ES(1501, 1), BF)
    spec.execute([ra, rb], res)
    torch.cuda.synchronize()
    st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    before = ja.ja_launch_count()
    with torch.cuda.graph(g, stream=st):
        spec.execute([ra, rb], res)
    assert ja.ja_launch_count() - before == 2      # the copy and the product, as outside
    for _ in range(2):
        res.payload.fill_(float("nan"))
        torch.cuda.current_stream().synchronize()
        g.replay()
        _check(res, a, b, BF)


def _drops_to(held):
    """Graphs are destroyed by the driver in its own time."""
    torch.cuda.synchronize()
    for _ in range(500):
        if ja.ja_debug_scratch_bytes() <= held:
            return True
        time.sleep(0.02)
    return False


def test_graph_outlives_its_spec():
    """The scratch that a graph recorded is the graph's as well: not handed to the next plan, and given back when the graph goes."""
    held = ja.ja_debug_scratch_bytes()
    a, b, ra, rb, res, spec = _problem(ES(1000, 1), ES(2001, 1), ES(1501, 1), BF)
    spec.execute([ra, rb], res)
    torch.cuda.synchronize()
    st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        spec.execute([ra, rb], res)
        spec.execute([ra, rb], res)
    mine = ja.ja_debug_scratch_bytes() - held
    assert mine > 0
    spec.close()
    assert ja.ja_debug_scratch_bytes() == held + mine
    a2, b2, ra2, rb2, res2, spec2 = _problem(ES(1000, 1), ES(2001, 1), ES(1501, 1), BF)
    a2, rb2 = -a2, upload(-b2, [ES(2001, 1), ES(1501, 1)])
    spec2.execute([ra2, rb2], res2)
    assert ja.ja_debug_scratch_bytes() == held + 2 * mine
    res.payload.fill_(float("nan"))
    g.replay()
    _check(res, a, b, BF)
    spec2.execute([ra2, rb2], res2)
    _check(res2, a2, b2, BF)
    spec2.close()
    g.replay()                                     # under way when the graph goes
    del g
    assert _drops_to(held)
    _check(res, a, b, BF)


def test_spec_dropped_while_a_capture_runs_and_with_its_work_under_way():
    held = ja.ja_debug_scratch_bytes()
    a, b, ra, rb, res, spec = _problem(ES(1000, 1), ES(2001, 1), ES(1501, 1), BF)
    a2, b2, ra2, rb2, res2, dropped = _problem(ES(1300, 2), ES(1501, 1), ES(1401, 3), BF)
    spec.execute([ra, rb], res)
    dropped.execute([ra2, rb2], res2)
    torch.cuda.synchronize()
    res2.payload.fill_(float("nan"))
    torch.cuda.current_stream().synchronize()
    other, st, g = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        spec.execute([ra, rb], res)
        with torch.cuda.stream(other):
            torch.cuda._sleep(200_000_000)
            dropped.execute([ra2, rb2], res2)
        both = ja.ja_debug_scratch_bytes()
        dropped.close()
        assert ja.ja_debug_scratch_bytes() == both          # its work has not ended
    res.payload.fill_(float("nan"))
    g.replay()
    _check(res, a, b, BF)
    _check(res2, a2, b2, BF)
    spec.close()
    del g
    assert _drops_to(held)


@pytest.mark.parametrize("ti,tj,tk", [(ES(1000, 1), ES(2001, 1), ES(1501, 1)), ([0, 100, 1301], [0, 130, 1931], [0, 135, 271, 1400]),
                                      (ES(1640, 3), list(range(0, 1407, 7)), ES(1520, 2)), (ES(65, 5), ES(3999, 1), ES(3000, 5))])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_values_that_are_not_finite_stay_in_their_row_and_column(ti, tj, tk, dtype):
    """and what lies between the blocks of a payload reaches no cell."""
    a, b, ra, rb, res, spec = _problem(ti, tj, tk, dtype)
    for x, r in ((a, ra), (b, rb)):
        between = torch.from_numpy(blocked.pack(np.ones(x.shape, np.uint16), r.splits) == 0).cuda()
        r.payload[:between.numel()][between] = float("nan")
    before = ja.ja_launch_count()
    spec.execute([ra, rb], res)
    assert ja.ja_launch_count() - before >= 2
    _check(res, a, b, dtype)
    a[5, 17], b[9, 33], b[tj[-1] - 1, 40], a[11, tj[-1] - 1] = float("inf"), float("nan"), float("-inf"), float("nan")
    ra, rb = upload(a, [ti, tj]), upload(b, [tj, tk])
    spec.execute([ra, rb], res)
    got = download(res)
    with np.errstate(invalid="ignore"):
        ref = si.to_f64(a) @ si.to_f64(b)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    ok = np.isfinite(ref)
    assert relfro(got[ok], ref[ok]) <= TOL[dtype] and np.array_equal(np.sign(got[np.isinf(ref)]), np.sign(ref[np.isinf(ref)]))

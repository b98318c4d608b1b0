"""Attention over sequences and blocks that are no whole pairs of 128-row tiles, on the tensor-memory kernel (its ragged form)
against the oracle. Lengths sit at the edges of tiles (128 rows), of pairs, of the 16-key groups of the P V product and of the
pieces a tile is made of. Tolerances: those of the other attention tests (ten half-ulps of the stored type). lse is held in f32:
scores of order five to 2^-21, exponentials to 2^-22, sums and a logarithm in f32 stay below 1e-5; where lengths are whole pairs of tiles
and blocks whole tiles a quarter of the exponentials are a cubic (7.5e-5 relative, so at most as much in a logarithm): 1e-4."""
import math

import numpy as np
import pytest
import torch

import paper_2609_03905_b200 as ja
import synth_inputs as si
from oracle import blocked, operators

from gpu_util import TOL, check_status, download, empty_like_tiling, relfro, upload

pytestmark = pytest.mark.gpu
ES = blocked.equal_splits
BF, F32, F16 = torch.bfloat16, torch.float32, torch.float16


def _run(B, S, Hq, Hkv, q_split, k_split, ends, causal, dtype, lse=False, b_blocks=None, g_split=None, scale=1.0 / math.sqrt(128)):
    grp = Hq // Hkv
    Q, K, V = (si.normal((B, S, h, 128), 0.0, 1.0, dtype, 4, 60 + n) for n, h in enumerate((Hq, Hkv, Hkv)))
    b_sp, g_sp = ES(B, b_blocks or B), g_split or ES(Hkv, max(1, Hkv // 2))
    h_sp = [grp * v for v in g_sp]
    d = [0, 128]
    rq, rk, rv = upload(Q, [b_sp, q_split, h_sp, d]), upload(K, [b_sp, k_split, g_sp, d]), upload(V, [b_sp, k_split, g_sp, d])
    ro = empty_like_tiling([B, S, Hq, 128], [b_sp, q_split, h_sp, d], dtype, fill=float("nan"))
    rl = empty_like_tiling([B, S, Hq], [b_sp, q_split, h_sp], F32, fill=float("nan")) if lse else None
    parts = {"b": b_sp, "q": q_split, "h": h_sp, "d": d, "k": k_split}
    if grp > 1:
        parts["g"] = g_sp
    spec = ja.Spec("bqhd,bkgd,bkgd->bqhd" if grp > 1 else "bqhd,bkhd,bkhd->bqhd", parts, "attention",
                   (scale, 1.0 if causal else 0.0) + tuple(float(e) for e in ends), "online_softmax")
    spec.execute([rq, rk, rv], [ro, rl] if lse else ro)
    got = download(ro)
    ref = operators.attention_gqa_packed(si.to_f64(Q), si.to_f64(K), si.to_f64(V), grp, ends or None, causal, {BF: "bf16", F16: "f16"}[dtype], scale)
    assert relfro(got, ref) <= TOL[dtype]
    # no row is worse than the whole: a row that lost or gained a key would be
    err = np.linalg.norm(got - ref, axis=-1) / np.maximum(np.linalg.norm(ref, axis=-1), 1e-3)
    assert err.max() <= 4 * TOL[dtype]
    if lse:
        whole = all(e % 256 == 0 for e in ends or [S]) and all(x % 128 == 0 for x in q_split + k_split)
        s0 = 0
        L = download(rl)
        for s1 in ends or [S]:
            K2 = np.repeat(si.to_f64(K)[:, s0:s1], grp, axis=2)
            want = operators.attention_lse(si.to_f64(Q)[:, s0:s1], K2, causal, scale)
            assert np.abs(L[:, s0:s1] - want).max() <= (1e-4 if whole and scale > 0 else 1e-5)
            s0 = s1
    check_status()


@pytest.mark.parametrize("S", [46, 63, 65, 127, 128, 129, 143, 145, 255, 257, 383, 384, 385, 641])
@pytest.mark.parametrize("causal", [True, False])
def test_one_block_of_any_length(S, causal):
    _run(2, S, 4, 4, [0, S], [0, S], [], causal, BF, lse=True)


@pytest.mark.parametrize("cut", [200, 125, 64, 72, 40, 96])     # 8-, 1-, 64-, 8-, 8- and 32-row pieces
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_short_blocks(cut, causal, dtype):
    S = cut * 6
    _run(2, S, 8, 2, ES(S, 6), ES(S, 6), [], causal, dtype, b_blocks=1)


@pytest.mark.parametrize("ends", [[50, 131, 400], [128, 256, 384], [64, 320, 1000], [777, 778, 1000], [1000]])
@pytest.mark.parametrize("causal,lse", [(True, False), (True, True), (False, False)])
def test_packed_sequences(ends, causal, lse):
    S = ends[-1]
    _run(2, S, 8, 4, [0] + ends, [0] + ends, ends, causal, BF, lse=lse)


# equal blocks with a shorter last one, several head blocks: the rows of a head block after the first start where the SHORT block
# says (download() looks at the guard zones)
@pytest.mark.parametrize("split,packed", [([0, 128, 256, 300], False), ([0, 300, 500], True), ([0, 777, 1291], True), ([0, 602, 668], True),
                                          ([0, 256, 384], False), ([0, 512, 768], False), ([0, 256, 384], True)])
@pytest.mark.parametrize("causal,lse", [(True, False), (False, True)])
@pytest.mark.parametrize("dtype,b_blocks", [(BF, 2), (F16, 1)])
def test_shorter_last_block(split, packed, causal, lse, dtype, b_blocks):
    S = split[-1]
    _run(2, S, 8, 4, split, split, split[1:] if packed else [], causal, dtype, lse=lse, b_blocks=b_blocks)


# a shorter last head block: its rows are shorter, so the kernels that hold rows of one length leave it to the mma.sync form
@pytest.mark.parametrize("S", [300, 256])
def test_shorter_last_head_block(S):
    _run(1, S, 3, 3, [0, S], [0, S], [], True, BF, lse=True, g_split=[0, 2, 3])
    _run(1, S, 6, 3, [0, S], [0, S], [], False, F16, g_split=[0, 2, 3])


# any scale: 0 (every key counts alike), a negative one (the most negative product wins)
@pytest.mark.parametrize("scale", [0.0, -1.0 / math.sqrt(128)])
@pytest.mark.parametrize("S,causal", [(300, True), (145, False), (512, True), (256, False)])
def test_scales_that_are_not_positive(S, causal, scale):
    _run(2, S, 4, 2, [0, S], [0, S], [], causal, BF if S % 2 else F16, lse=True, scale=scale)


@pytest.mark.parametrize("split", [[0, 300], [0, 37, 101, 200, 333], [0, 200, 400]])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_later_values_that_are_not_finite(split, bad):
    """V is NaN or infinite from some key on: no query more than 63 positions before it notices (causal; half a key tile)."""
    S, H = split[-1], 2
    Q, K, V = (si.normal((1, S, H, 128), 0.0, 1.0, BF, 4, 100 + n) for n in range(3))
    ref = operators.attention_gqa_packed(si.to_f64(Q), si.to_f64(K), si.to_f64(V), 1, None, True, "bf16")
    sp = [[0, 1], split, [0, H], [0, 128]]
    spec = ja.Spec("bqhd,bkhd,bkhd->bqhd", {"b": sp[0], "q": sp[1], "h": sp[2], "d": sp[3], "k": sp[1]}, "attention", (1.0 / math.sqrt(128), 1.0),
                   "online_softmax")
    for first_bad in (100, 190, 127, 128, 250, S - 1):
        V2 = V.clone()
        V2[:, first_bad:] = bad
        ro = empty_like_tiling([1, S, H, 128], sp, BF, fill=float("nan"))
        spec.execute([upload(Q, sp), upload(K, sp), upload(V2, sp)], ro)
        got = download(ro)
        check_status()
        n = first_bad - 63
        assert relfro(got[:, :n], ref[:, :n]) <= TOL[BF]
        assert not np.isfinite(got[:, first_bad:]).any()


@pytest.mark.parametrize("S", [131, 145, 300, 512, 768])        # ragged lengths and whole pairs of tiles
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_scores_of_minus_infinity(S, causal, dtype):
    """The first 130 keys score -inf with every query (more than a key tile): a row's weights are those of its other keys, whose scores
    lie far below 0 here, and a row without any has O = 0 and lse = -inf."""
    H, n = 2, 130
    Q, K, V = (si.normal((1, S, H, 128), 0.0, 1.0, dtype, 4, 90 + i) for i in range(3))
    Q[..., 0] = 1.0
    K[:, n:, :, 0] = -300.0
    ref = operators.attention(si.to_f64(Q)[:, n:], si.to_f64(K)[:, n:], si.to_f64(V)[:, n:], causal, {BF: "bf16", F16: "f16"}[dtype])
    ref_l = operators.attention_lse(si.to_f64(Q)[:, n:], si.to_f64(K)[:, n:], causal)
    K[:, :n, :, 0] = float("-inf")
    sp = [[0, 1], [0, S], ES(H, 2), [0, 128]]
    ro, rl = empty_like_tiling([1, S, H, 128], sp, dtype, fill=float("nan")), empty_like_tiling([1, S, H], sp[:3], F32, fill=float("nan"))
    ja.Spec("bqhd,bkhd,bkhd->bqhd", {"b": sp[0], "q": sp[1], "h": sp[2], "d": sp[3], "k": sp[1]}, "attention",
            (1.0 / math.sqrt(128), 1.0 if causal else 0.0), "online_softmax").execute([upload(Q, sp), upload(K, sp), upload(V, sp)], [ro, rl])
    got, lse = download(ro), download(rl)
    check_status()
    assert relfro(got[:, n:], ref) <= TOL[dtype]
    assert np.abs(lse[:, n:] - ref_l).max() <= 1e-4     # logarithms of order 30
    if causal:
        assert (got[:, :n] == 0).all() and np.isneginf(lse[:, :n]).all()


def test_queries_and_keys_cut_differently():
    S = 600
    _run(1, S, 4, 2, [0, 130, 391, 600], ES(S, 3), [], True, BF)
    _run(1, S, 4, 4, ES(S, 4), [0, 64, 512, 600], [], True, F16, lse=True)


def test_nothing_leaks_from_other_sequences():
    """Keys and values of the second sequence are infinite: the first one's results must not notice."""
    ends, S, H = [77, 200], 200, 2
    Q, K, V = (si.normal((1, S, H, 128), 0.0, 1.0, BF, 4, 70 + n) for n in range(3))
    ref = operators.attention_gqa_packed(si.to_f64(Q), si.to_f64(K), si.to_f64(V), 1, ends, True, "bf16")
    K[:, 77:] = float("inf")
    V[:, 77:] = float("nan")
    sp = [[0, 1], [0] + ends, [0, H], [0, 128]]
    ro = empty_like_tiling([1, S, H, 128], sp, BF)
    ja.Spec("bqhd,bkhd,bkhd->bqhd", {"b": sp[0], "q": sp[1], "h": sp[2], "d": sp[3], "k": sp[1]}, "attention",
            (1.0 / math.sqrt(128), 1.0, 77.0, 200.0), "online_softmax").execute([upload(Q, sp), upload(K, sp), upload(V, sp)], ro)
    torch.cuda.synchronize()
    payload = ro.payload[: 77 * H * 128].reshape(1, 77, H, 128).to(torch.float64).cpu().numpy()
    assert relfro(payload, ref[:, :77]) <= TOL[BF]
    check_status()


def test_more_items_than_a_wave_and_a_graph_replay():
    S = 300
    Q, K, V = (si.normal((8, S, 32, 128), 0.0, 1.0, BF, 4, 80 + n) for n in range(3))
    sp = [ES(8, 8), [0, S], ES(32, 4), [0, 128]]
    rels = [upload(x, sp) for x in (Q, K, V)]
    ro = empty_like_tiling([8, S, 32, 128], sp, BF, fill=float("nan"))
    spec = ja.Spec("bqhd,bkhd,bkhd->bqhd", {"b": sp[0], "q": sp[1], "h": sp[2], "d": sp[3], "k": sp[1]}, "attention", (1.0 / math.sqrt(128), 1.0),
                   "online_softmax")
    spec.execute(rels, ro)
    ref = operators.attention_gqa_packed(si.to_f64(Q), si.to_f64(K), si.to_f64(V), 1, None, True, "bf16")
    first = download(ro)
    assert relfro(first, ref) <= TOL[BF]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        spec.execute(rels, ro)
    ro.payload.fill_(float("nan"))
    g.replay()
    g.replay()
    assert np.array_equal(download(ro), first)
    check_status()

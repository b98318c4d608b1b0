"""f32 contractions under any tiling and index order (k_contract_f32.cu) and the general join-agg (k_generic.cu) against fp64
numpy. f32 sums of up to a few thousand products of order one: 2^-24 per rounding, well inside 1e-5 relative; MAX is exact."""
import numpy as np
import pytest
import torch

import paper_2609_03905_b200 as ja
import synth_inputs as si
from oracle import blocked

from gpu_util import TOL, check_status, download, empty_like_tiling, relfro, upload

pytestmark = pytest.mark.gpu
ES = blocked.equal_splits
BF, F32, F16 = torch.bfloat16, torch.float32, torch.float16


def _run(einsum, cuts, fn, agg, dtypes, out_dtype, ref):
    ins, out = einsum.split("->")
    ext = {c: s[-1] for c, s in cuts.items()}
    dense = [si.normal(tuple(ext[c] for c in t), 0.0, 1.0, dt, 33, 40 + n) for n, (t, dt) in enumerate(zip(ins.split(","), dtypes))]
    rels = [upload(d, [cuts[c] for c in t]) for d, t in zip(dense, ins.split(","))]
    res = empty_like_tiling([ext[c] for c in out], [cuts[c] for c in out], out_dtype, fill=float("nan"))
    ja.Spec(einsum, cuts, fn, (), agg).execute(rels, res)
    got = download(res)
    check_status()
    want = ref(*[si.to_f64(d) for d in dense])
    if agg == "max":
        assert np.array_equal(got, want)
    else:
        assert relfro(got, want) <= TOL[out_dtype]
        assert np.abs(got - want).max() <= {F32: 2.0 ** -14, BF: 2.0 ** -7, F16: 2.0 ** -10}[out_dtype] * np.abs(want).max()


def _product(einsum, cuts, out_dtype=F32):
    _run(einsum, cuts, "mul", "sum", (F32, F32), out_dtype, lambda a, b: np.einsum(einsum, a, b))


@pytest.mark.parametrize("einsum", ["ij,jk->ik", "ij,kj->ik", "ji,jk->ik", "ji,kj->ki", "ij,jk->ki", "bij,bjk->bik", "bij,bkj->bik", "bji,bjk->bik", "ibj,bjk->bik",
                                    "bij,jk->bik", "abij,abkj->abik", "bij,bjk->ikb"])
@pytest.mark.parametrize("cut", [1, 3])
def test_index_orders(einsum, cut):
    ext = {"a": 2, "b": 3, "i": 40, "j": 52, "k": 36}
    _product(einsum, {c: ES(ext[c], min(cut, ext[c])) for c in set(einsum) - set(",->")})


@pytest.mark.parametrize("einsum", ["ij,jk->ik", "ij,kj->ik", "ji,jk->ik", "ji,kj->ik"])
@pytest.mark.parametrize("m,k,n,cut", [
    (1, 1, 1, 1), (31, 33, 65, 1), (128, 64, 128, 2), (260, 497, 270, 4), (64, 4096, 64, 2),     # the last: slices of the contracted index
    (1700, 36, 1500, 1), (1536, 40, 1664, 2),                                                   # 64- and 128-wide tiles
    (1601, 70, 1501, 3),                                                                        # ragged, odd
])
def test_tilings(einsum, m, k, n, cut):
    out = BF if m == 260 and einsum != "ij,jk->ik" else F32
    _product(einsum, {"i": ES(m, cut), "j": ES(k, cut), "k": ES(n, cut)}, out)


@pytest.mark.parametrize("einsum,fn,agg,ref", [
    ("ij,j->i", "mul", "sum", lambda a, b: a @ b),
    ("bij->bj", "ident", "max", lambda a: a.max(1)),
    ("bij->b", "square", "sum", lambda a: (a * a).sum((1, 2))),
    ("bij->i", "ident", "sum", lambda a: a.sum((0, 2))),
    ("bij->j", "ident", "max", lambda a: a.max((0, 1))),
    ("bij->ji", "ident", "sum", lambda a: a.sum(0).T),
    ("i,k->ik", "mul", "none", lambda a, b: np.outer(a, b)),
    ("ij,ij->j", "mul", "sum", lambda a, b: (a * b).sum(0)),
    ("ij,ji->i", "add", "max", lambda a, b: (a + b.T).max(1)),
    ("bij,bij->b", "mul", "sum", lambda a, b: (a * b).sum((1, 2))),
    ("ij,jk,k->i", "mul", "sum", lambda a, b, c: a @ b @ c),
    ("i,ij,j,jk->k", "mul", "sum", lambda a, b, c, d: ((a @ b) * c) @ d),
])
@pytest.mark.parametrize("sizes,cut", [((2, 32, 32, 8), 1), ((3, 61, 47, 29), 4), ((5, 130, 257, 33), 3), ((2, 7, 1, 3), 1)])
@pytest.mark.parametrize("dtype", [F32, BF])
def test_general_join_agg(einsum, fn, agg, ref, sizes, cut, dtype):
    ins = einsum.split("->")[0].split(",")
    ext = dict(zip("bijk", sizes))
    cuts = {c: ES(ext[c], min(cut, ext[c])) for c in set(einsum) - set(",->")}
    if agg == "max" and fn == "add":   # a sum of two cells is rounded: exact only against the same f32 sum
        ref32 = lambda a, b: (a.astype(np.float32) + b.astype(np.float32).T).max(1).astype(np.float64)
        return _run(einsum, cuts, fn, agg, [dtype] * len(ins), F32, ref32)
    _run(einsum, cuts, fn, agg, [dtype] * len(ins), dtype if agg == "max" else F32, ref)


def test_a_long_reduction_over_a_cluster():
    _run("bij->b", {"b": ES(2, 2), "i": ES(500, 4), "j": ES(511, 2)}, "square", "sum", (BF,), F32, lambda a: (a * a).sum((1, 2)))
    _run("ij,j->i", {"i": ES(3, 1), "j": ES(100003, 7)}, "mul", "sum", (F32, F32), F32, lambda a, b: a @ b)


def test_maximum_keeps_infinities():
    x = torch.full((3, 70), float("-inf"))
    x[1, 5] = float("inf")
    cuts = {"i": ES(3, 1), "j": ES(70, 3)}
    r, out = upload(x, [cuts["i"], cuts["j"]]), empty_like_tiling([70], [cuts["j"]], F32, fill=float("nan"))
    ja.Spec("ij->j", cuts, "ident", (), "max").execute([r], out)
    assert np.array_equal(download(out), x.max(0).values.double().numpy())
    check_status()


def test_a_block_of_more_than_2_to_31_bytes_after_the_summed_index():
    """Two slices of 2 GiB in one block: the step from a cell to the next one of the sum does not fit 32 bits. a + b is one rounding."""
    n = 16384 * 32768
    cuts = {"k": [0, 2], "i": [0, 16384], "j": [0, 32768]}
    x = ja.Relation([2, 16384, 32768], [cuts[c] for c in "kij"], F32, torch.randn(2 * n, device="cuda"))
    out = ja.Relation([16384, 32768], [cuts[c] for c in "ij"], F32, torch.full((n,), float("nan"), device="cuda"))
    ja.Spec("kij->ij", cuts, "ident", (), "sum").execute([x], out)
    assert torch.equal(out.payload, x.payload[:n] + x.payload[n:])
    check_status()


def test_an_index_of_more_than_2_to_30_cells():
    """Equal intervals with a shorter last one on an index whose interval ends leave 31 bits: the form with 64-bit coordinates."""
    n = (1 << 30) + 64
    cuts = {"i": [0, 2], "j": [0, 1 << 30, n]}
    x = ja.Relation([2, n], [cuts["i"], cuts["j"]], BF)
    x.payload.normal_()
    out = ja.Relation([n], [cuts["j"]], F32, torch.full((n,), float("nan"), device="cuda"))
    ja.Spec("ij->j", cuts, "ident", (), "sum").execute([x], out)
    check_status()
    for lo, hi, at in ((0, 1 << 30, 0), (1 << 30, n, 2 << 30)):       # the two blocks: [2, 2^30] cells, then [2, 64]
        w = hi - lo
        assert torch.equal(out.payload[lo:hi], x.payload[at: at + w].float() + x.payload[at + w: at + 2 * w].float())


# a queue of products, each of the one before it: launches that let the next one in at their start, and ones that do not (32 x 32 tiles:
# 296 to 444 at four CTAs an SM, 222 to 296 at three)
@pytest.mark.parametrize("b,cut", [(60, 1), (74, 1), (80, 1), (111, 1), (112, 1), (55, 2), (60, 2), (75, 2)])
def test_queue_of_products(b, cut):
    n = 61
    sb, sn = ES(b, 1), ES(n, cut)
    x = si.normal((b, n, n), 0.0, 1.0, F32, 33, 50)
    w = (si.normal((b, n, n), 0.0, 1.0, F32, 33, 51) * n ** -0.5).contiguous()
    cur, rw = upload(x, [sb, sn, sn]), upload(w, [sb, sn, sn])
    spec = ja.Spec("bij,bjk->bik", {"b": sb, "i": sn, "j": sn, "k": sn})
    steps = [cur] + [empty_like_tiling([b, n, n], [sb, sn, sn], F32, fill=float("nan")) for _ in range(6)]
    for _ in range(2):
        for s, d in zip(steps, steps[1:]):
            spec.execute([s, rw], d)
    want = si.to_f64(x)
    for _ in range(6):
        want = want @ si.to_f64(w)
    got = download(steps[-1])
    check_status()
    assert relfro(got, want) <= 6 * TOL[F32]

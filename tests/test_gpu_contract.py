"""Tensor-core contractions under any tiling and index order (k_contract_tc.cu) against an fp64 einsum of the same 16-bit
inputs. Tolerances: ten half-ulps of the stored type (gpu_util.TOL); f32 outputs 2e-6 relative, the size of f32 sums of up to
a few hundred products (2^-24 per rounding, tens of roundings)."""
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


def _run(einsum, cuts, dtype, out_dtype):
    """cuts: letter -> split points."""
    ins, out = einsum.split("->")
    ext = {c: s[-1] for c, s in cuts.items()}
    dense = [si.normal(tuple(ext[c] for c in t), 0.0, 1.0, dtype, 31, 40 + n) for n, t in enumerate(ins.split(","))]
    rels = [upload(d, [cuts[c] for c in t]) for d, t in zip(dense, ins.split(","))]
    res = empty_like_tiling([ext[c] for c in out], [cuts[c] for c in out], out_dtype, fill=float("nan"))
    ja.Spec(einsum, cuts, "mul", (), "sum").execute(rels, res)
    got = download(res)
    check_status()
    ref = np.einsum(einsum, *[si.to_f64(d) for d in dense])
    assert relfro(got, ref) <= (2e-6 if out_dtype == F32 else TOL[out_dtype]), einsum
    ulp = 2.0 ** {BF: -7, F16: -10, F32: -17}[out_dtype]      # of the largest value: a misplaced cell is far outside it
    assert np.abs(got - ref).max() <= ulp * np.abs(ref).max()


# every order of the indices: contiguous index contracted or not in either operand, batch index first, in the middle, in one
# operand only, last in the output; two batch indices
@pytest.mark.parametrize("einsum", ["bij,bjk->bik", "bij,bkj->bik", "bji,bjk->bik", "bji,bkj->bik", "ij,kj->ik", "ji,jk->ik", "ji,kj->ki", "ij,jk->ki",
                                    "ibj,bjk->bik", "bij,jk->bik", "ij,bkj->bik", "abij,abkj->abik", "bij,bjk->ikb", "jbi,kbj->ibk"])
@pytest.mark.parametrize("cut", [1, 3])
def test_index_orders(einsum, cut):
    ext = {"a": 2, "b": 3, "i": 144, "j": 72, "k": 136}
    _run(einsum, {c: ES(ext[c], min(cut, ext[c])) for c in set(einsum) - set(",->")}, BF, BF)


# every piece width of the loaders (8, 4, 2, 1 cells: common divisor of the contiguous index's split points), equal and ragged
# blocks, extents one off a tile or a stage, fewer rows than one piece
@pytest.mark.parametrize("einsum", ["ij,jk->ik", "bij,bkj->bik", "bji,bjk->bki"])
@pytest.mark.parametrize("si_,sj,sk", [
    (ES(128, 1), ES(64, 1), ES(64, 1)),                                  # one tile, one stage
    (ES(256, 2), ES(344, 2), ES(172, 1)),                                # 172-cell block rows: pieces of 4
    (ES(260, 2), ES(300, 2), ES(132, 2)),                                # 130, 150, 66: pieces of 2
    (ES(129, 1), ES(65, 1), ES(257, 1)),                                 # one past a tile / a stage
    ([0, 100, 301], [0, 130, 331], [0, 135, 271]),                       # ragged, odd
    ([0, 8, 24, 152], [0, 64, 72, 200], [0, 56, 64, 264]),               # ragged multiples of 8
    (ES(7, 1), ES(9, 1), ES(5, 1)),
    (list(range(20)), list(range(71)), list(range(34))),                 # every sub-tensor one cell
])
def test_tilings(einsum, si_, sj, sk):
    cuts = {"i": si_, "j": sj, "k": sk, "b": ES(2, 2)}
    _run(einsum, {c: s for c, s in cuts.items() if c in einsum}, BF, BF if einsum == "ij,jk->ik" else F32)   # that form wants one type


# split over a cluster (long contracted index, few tiles) with the columns or the rows short, f16, and a many-tile product
@pytest.mark.parametrize("m,k,n,gk", [(32, 4096, 520, 8), (40, 1472, 1141, 2), (520, 4096, 16, 1), (136, 2368, 276, 4), (1, 2048, 640, 1),
                                      (2050, 258, 1290, 3)])
@pytest.mark.parametrize("dtype,out", [(BF, BF), (F16, F16), (F16, F32)])
def test_sizes(m, k, n, gk, dtype, out):
    _run("ij,kj->ik", {"i": ES(m, 1), "j": ES(k, gk), "k": ES(n, 2)}, dtype, out)


def test_nothing_leaks_from_rows_that_do_not_exist():
    """Cells next to the operands' ends in memory are infinite: none of them may reach a result."""
    m, k, n = 130, 70, 66
    raw = torch.full((1 << 18,), float("inf"), dtype=BF, device="cuda")
    a, b = si.normal((m, k), 0.0, 1.0, BF, 31, 50), si.normal((k, n), 0.0, 1.0, BF, 31, 51)
    pa = raw[64 * 100: 64 * 100 + (m * k + 63) // 64 * 64]
    pb = raw[64 * 1000: 64 * 1000 + (k * n + 63) // 64 * 64]
    pa[: m * k].copy_(a.reshape(-1))
    pb[: k * n].copy_(b.reshape(-1))
    one = lambda e: [0, e]
    ra, rb = ja.Relation([m, k], [one(m), one(k)], BF, pa), ja.Relation([k, n], [one(k), one(n)], BF, pb)
    res = empty_like_tiling([m, n], [one(m), one(n)], BF)
    ja.Spec("ij,jk->ik", {"i": one(m), "j": one(k), "k": one(n)}, "mul", (), "sum").execute([ra, rb], res)
    assert relfro(download(res), si.to_f64(a) @ si.to_f64(b)) <= TOL[BF]
    check_status()


@pytest.mark.parametrize("K", [64, 200, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_an_f32_output_is_as_exact_as_f32_sums(K, dtype):
    """Products of 16-bit cells are exact in f32; the tensor core's sums of them may be no further from fp64 than adding them one after
    the other in f32 (a quarter more for the scatter of one sample)."""
    a, b = si.normal((2, 48, K), 0.0, 1.0, dtype, 31, 60), si.normal((2, 40, K), 0.0, 1.0, dtype, 31, 61)
    cuts = {"b": ES(2, 2), "i": ES(48, 1), "j": ES(K, 2), "k": ES(40, 1)}
    res = empty_like_tiling([2, 48, 40], [cuts[c] for c in "bik"], F32, fill=float("nan"))
    ja.Spec("bij,bkj->bik", cuts, "mul", (), "sum").execute([upload(a, [cuts[c] for c in "bij"]), upload(b, [cuts[c] for c in "bkj"])], res)
    a64, b64 = si.to_f64(a), si.to_f64(b)
    ref = np.einsum("bij,bkj->bik", a64, b64)
    one_by_one = np.zeros((2, 48, 40), np.float32)
    for j in range(K):
        one_by_one += (a64[:, :, None, j] * b64[:, None, :, j]).astype(np.float32)
    assert relfro(download(res), ref) <= 1.25 * relfro(one_by_one.astype(np.float64), ref)
    check_status()


# two-index products that TMA cannot address, on both sides of the line between the plain-ALU kernel and this one
@pytest.mark.parametrize("m,gi,k,gj,n,gk", [(64, 2, 314, 8, 320, 4), (250, 2, 313, 1, 333, 4), (16, 1, 700, 8, 320, 1), (64, 8, 1501, 64, 320, 4),
                                            (500, 2, 314, 8, 1007, 8), (33, 3, 70, 2, 75, 5)])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_products_in_odd_intervals(m, gi, k, gj, n, gk, dtype):
    _run("ij,jk->ik", {"i": ES(m, gi), "j": ES(k, gj), "k": ES(n, gk)}, dtype, dtype)

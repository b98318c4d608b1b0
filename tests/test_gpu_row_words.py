"""Row-structured join-aggs on widths and tilings whose rows start anywhere (aligned words with masked ends): rows of one cell,
runs shorter than a word, runs that start at every even offset, the longest row a CTA holds and one past it, infinities. Against
the oracle's formulas in fp64; MAX exact; tolerances of the other row tests (ten half-ulps of the stored type, 1e-5 for f32
statistics)."""
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
EPS = 1e-5

CASES = [((5, 1), ES(5, 1), ES(1, 1)), ((9, 7), ES(9, 2), ES(7, 3)), ((33, 139), ES(33, 4), ES(139, 4)), ((40, 903), ES(40, 3), [0, 1, 500, 903]),
         ((17, 13676), ES(17, 1), ES(13676, 1)), ((6, 16001), ES(6, 2), ES(16001, 8)), ((64, 3239), ES(64, 2), ES(3239, 1)),
         ((12, 96), [0, 5, 12], ES(96, 1)), ((50, 260), ES(50, 1), list(range(0, 261, 20))), ((3, 33001), ES(3, 1), ES(33001, 2)),
         ((21, 2000), ES(21, 2), [0, 1000, *range(1010, 2001, 10)]),       # more words than a CTA holds, counted by the widest run
         ((9, 800), ES(9, 1), [*range(0, 800, 3), 800]), ((9, 800), ES(9, 2), list(range(0, 801, 8))), ((9, 660), ES(9, 1), [0, 300, *range(309, 661, 9)])]


@pytest.mark.parametrize("shape,si_,sj", CASES)
@pytest.mark.parametrize("dtype", [BF, F16, F32])
def test_rmsnorm_forms(shape, si_, sj, dtype):
    x, g = si.normal(shape, 0.0, 2.0, dtype, 38, 1), si.normal((shape[1],), 1.0, 0.1, dtype, 38, 2)
    x64, g64 = si.to_f64(x), si.to_f64(g)
    parts = {"i": si_, "j": sj}
    rx, rg = upload(x, [si_, sj]), upload(g, [sj])
    y, y2 = (empty_like_tiling([*shape], [si_, sj], dtype, fill=float("nan")) for _ in range(2))
    ss = empty_like_tiling([shape[0]], [si_], F32, fill=float("nan"))
    ja.Spec("ij,j->ij", parts, "rmsnorm", (EPS,), "none").execute([rx, rg], y)
    ja.Spec("ij->i", parts, "square", (), "sum").execute([rx], ss)
    ja.Spec("ij,i,j->ij", parts, "rms_scale", (EPS,), "none").execute([rx, ss, rg], y2)
    want = x64 / np.sqrt((x64 ** 2).mean(1, keepdims=True) + EPS) * g64
    assert relfro(download(ss), (x64 ** 2).sum(1)) <= TOL[F32]
    for r in (y, y2):
        assert relfro(download(r), want) <= TOL[dtype]
    check_status()


@pytest.mark.parametrize("shape,si_,sj", CASES)
@pytest.mark.parametrize("dtype", [BF, F16, F32])
def test_softmax_forms(shape, si_, sj, dtype):
    x = si.normal((2, *shape), 0.0, 2.0, dtype, 38, 3)
    x64 = si.to_f64(x)
    hs = ES(2, 2)
    parts, sp = {"h": hs, "i": si_, "j": sj}, [hs, si_, sj]
    rx = upload(x, sp)
    y, y2 = (empty_like_tiling([2, *shape], sp, dtype, fill=float("nan")) for _ in range(2))
    m, l = (empty_like_tiling([2, shape[0]], sp[:2], F32, fill=float("nan")) for _ in range(2))
    ja.Spec("hij->hij", parts, "softmax", (), "none").execute([rx], y)
    ja.Spec("hij->hi", parts, "ident", (), "max").execute([rx], m)
    ja.Spec("hij,hi->hi", parts, "exp_sub", (), "sum").execute([rx, m], l)
    ja.Spec("hij,hi,hi->hij", parts, "exp_sub_div", (), "none").execute([rx, m, l], y2)
    mx = x64.max(-1)
    e = np.exp(x64 - mx[..., None])
    assert np.array_equal(download(m), mx)
    assert relfro(download(l), e.sum(-1)) <= TOL[F32]
    for r in (y, y2):
        assert relfro(download(r), e / e.sum(-1, keepdims=True)) <= TOL[dtype]
    check_status()


def test_softmax_with_masked_cells():
    """Cells of -inf, and of the type's lowest value, get probability zero; rows of other blocks never enter a row's sum."""
    x = torch.zeros(6, 45, dtype=F32)
    x[0, 3:] = float("-inf")
    x[1, ::2] = torch.finfo(F32).min
    x[2:] = 1e30
    sp = [ES(6, 2), ES(45, 4)]
    y = empty_like_tiling([6, 45], sp, F32)
    ja.Spec("ij->ij", {"i": sp[0], "j": sp[1]}, "softmax", (), "none").execute([upload(x, sp)], y)
    assert np.abs(download(y) - torch.softmax(x.double(), -1).numpy()).max() <= 1e-6
    check_status()

"""The TMA-fed matmul on row blocks that are no whole 128-row halves: pairs of CTAs whose two row tiles may lie in different
blocks, an odd number of row tiles, blocks shorter than a tile that do not divide it."""
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

ROWS = [(1260, 1), (600, 3), (500, 4), (272, 4), (1088, 2), (375, 3), (129, 1), (136, 1), (3 * 136, 3)]


def _operands(m, k, n, gi, gj, gk, dtype):
    A, B = si.normal((m, k), 0.0, 1.0, dtype, 35, 1), si.normal((k, n), 0.0, 0.05, dtype, 35, 2)
    ti, tj, tk = ES(m, gi), ES(k, gj), ES(n, gk)
    return si.to_f64(A), si.to_f64(B), upload(A, [ti, tj]), upload(B, [tj, tk]), ti, tj, tk


@pytest.mark.parametrize("m,gi", ROWS)
@pytest.mark.parametrize("k,n,gj,gk", [(512, 768, 2, 1), (256, 520, 1, 1), (768, 1376, 3, 2)])
@pytest.mark.parametrize("cta_group", [2, 1])
def test_matmul(m, gi, k, n, gj, gk, cta_group):
    ja.ja_debug_set("gemm_loader", 0)            # the TMA form even where the cp.async form would be chosen
    ja.ja_debug_set("gemm_cta_group", cta_group)
    a, b, ra, rb, ti, tj, tk = _operands(m, k, n, gi, gj, gk, BF)
    out = empty_like_tiling([m, n], [ti, tk], BF, fill=float("nan"))
    ja.Spec("ij,jk->ik", {"i": ti, "j": tj, "k": tk}).execute([ra, rb], out)
    ref = a @ b
    assert relfro(download(out), ref) <= TOL[BF]
    assert np.abs(download(out) - ref).max() <= 2.0 ** -7 * np.abs(ref).max()
    check_status()


@pytest.mark.parametrize("m,gi", [r for r in ROWS if r[0] // r[1] > 128])
def test_fused_add_and_join(m, gi):
    k, n = 512, 768
    a, b, ra, rb, ti, tj, tk = _operands(m, k, n, gi, 2, 3, F16)
    X = si.normal((m, n), 0.0, 1.0, F16, 35, 3)
    out = empty_like_tiling([m, n], [ti, tk], F16, fill=float("nan"))
    ja.Spec("ij,jk,ik->ik", {"i": ti, "j": tj, "k": tk}, "matmul_add", (), "sum").execute([ra, rb, upload(X, [ti, tk])], out)
    assert relfro(download(out), a @ b + si.to_f64(X)) <= TOL[F16]
    check_status()


@pytest.mark.parametrize("m,gi", ROWS)
def test_join_only(m, gi):
    k, n, gj = 512, 512, 4
    a, b, ra, rb, ti, tj, tk = _operands(m, k, n, gi, gj, 2, BF)
    parts = empty_like_tiling([gj, m, n], [list(range(gj + 1)), ti, tk], BF, fill=float("nan"))
    ja.Spec("ij,jk->ik", {"i": ti, "j": tj, "k": tk}).execute_join([ra, rb], parts)
    got = download(parts)
    for c in range(gj):
        assert relfro(got[c], a[:, tj[c]:tj[c + 1]] @ b[tj[c]:tj[c + 1]]) <= TOL[BF]
    check_status()

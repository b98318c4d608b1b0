"""Products that leave most of the chip idle as whole tiles: few rows against a large second operand (k_stream_tc.cu), and few tiles, or a few
in the last round, split along the contracted index over clusters (k_gemm_tc.cu), against an fp64 product of the same 16-bit inputs.
Tolerance: gpu_util.TOL, ten half-ulps of the stored type."""
import os
import subprocess
import sys

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


# few rows that need no copy: row blocks of any height, column tiles inside blocks and across them, every number of slices
@pytest.mark.parametrize("m,gi,k,gj,n,gk", [(32, 1, 4096, 8, 11008, 8), (8, 1, 512, 1, 256, 1), (1, 1, 2048, 2, 4096, 4), (100, 1, 1024, 4, 1000, 1), (128, 4, 2048, 1, 640, 5),
                                            (36, 3, 1024, 1, 768, 1), (64, 1, 64, 1, 8192, 1), (16, 2, 4096, 1, 1504, 1)])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_few_rows(m, gi, k, gj, n, gk, dtype):
    a, b, ra, rb, res, spec = _problem(ES(m, gi), ES(k, gj), ES(n, gk), dtype)
    spec.execute([ra, rb], res)
    _check(res, a, b, dtype)


# whole tiles, split tiles, and both: few tiles (clusters of two and of four pairs), one more than a round, blocks whose ends are inside a slice
@pytest.mark.parametrize("m,gi,k,gj,n,gk", [(512, 4, 4096, 8, 1024, 8), (1024, 8, 4096, 8, 2048, 4), (256, 2, 2048, 2, 4096, 8), (1280, 1, 1024, 1, 3840, 1),
                                            (600, 1, 1376, 8, 512, 1), (2560, 10, 512, 1, 1920, 1)])
@pytest.mark.parametrize("fn", ["mul", "matmul_add", "swiglu_up", "matmul_rope"])
@pytest.mark.parametrize("dtype", [BF, F16])
def test_split_tiles(m, gi, k, gj, n, gk, fn, dtype):
    ti, tj, tk = ES(m, gi), ES(k, gj), ES(n, gk)
    if fn != "mul" and ((n // gk) % 128 or (k // gj) % 8):
        pytest.skip("the fused forms take whole 128-column blocks and rows of whole 16 bytes")
    a, b, ra, rb, res, spec = _problem(ti, tj, tk, dtype)
    parts, scale = {"i": ti, "j": tj, "k": tk}, k ** -0.5
    b = (b.float() * scale).to(dtype)
    rb = upload(b, [tj, tk])
    ref = si.to_f64(a) @ si.to_f64(b)
    if fn == "mul":
        spec.execute([ra, rb], res)
    elif fn == "matmul_add":
        x = si.normal((m, n), 0.0, 1.0, dtype, 37, 42)
        ref = ref + si.to_f64(x)
        ja.Spec("ij,jk,ik->ik", parts, fn).execute([ra, rb, upload(x, [ti, tk])], res)
    elif fn == "swiglu_up":
        b2 = (si.normal((k, n), 0.0, 1.0, dtype, 37, 43).float() * scale).to(dtype)
        ref = ref / (1.0 + np.exp(-ref)) * (si.to_f64(a) @ si.to_f64(b2))
        ja.Spec("ij,jk,jk->ik", parts, fn).execute([ra, rb, upload(b2, [tj, tk])], res)
    else:
        s_len, d = m // 2, 128
        ang = np.arange(s_len)[:, None] * 10000.0 ** (-2.0 * np.arange(d // 2) / d)[None, :]
        c, s = np.tile(np.cos(ang), (2, n // d)), np.tile(np.sin(ang), (2, n // d))
        x0, x1 = ref[:, 0::2].copy(), ref[:, 1::2].copy()
        ref[:, 0::2], ref[:, 1::2] = x0 * c - x1 * s, x0 * s + x1 * c
        ja.Spec("ij,jk->ik", parts, fn, (10000.0, float(s_len), float(d))).execute([ra, rb], res)
    got = download(res)
    check_status()
    assert relfro(got, ref) <= TOL[dtype]
    assert np.abs(got - ref).max() <= 2.0 ** (-6 if dtype == BF else -9) * np.abs(ref).max()


# the join alone over ONE contracted block: few tiles, which as an aggregated product would be split, in partial relations of both cell sizes
@pytest.mark.parametrize("m,gi,k,n,gk", [(256, 1, 4096, 4096, 1), (512, 4, 4096, 1024, 2), (384, 3, 2048, 768, 3)])
@pytest.mark.parametrize("dtype,pdtype", [(BF, torch.float32), (F16, torch.float32), (BF, BF), (F16, F16)])
def test_join_only_one_copy(m, gi, k, n, gk, dtype, pdtype):
    ti, tj, tk = ES(m, gi), ES(k, 1), ES(n, gk)
    a, b, ra, rb, _, spec = _problem(ti, tj, tk, dtype)
    part = empty_like_tiling([1, m, n], [[0, 1], ti, tk], pdtype, fill=float("nan"))
    spec.execute_join([ra, rb], part)
    got, ref = download(part)[0], si.to_f64(a) @ si.to_f64(b)
    check_status()
    # in f32 the tensor core's truncated sums show: one unit of 2^-23 of the running sum for each of k / 16 additions, at most
    assert relfro(got, ref) <= (k / 16 * 2.0 ** -23 if pdtype == torch.float32 else TOL[dtype])


FIRST_PLANS = """
import sys
import torch
import paper_2609_03905_b200 as ja
from oracle import blocked
ES = blocked.equal_splits
for name in sys.argv[1:]:
    dt, ti = {"f16": (torch.float16, ES(2560, 1)), "bf16": (torch.bfloat16, ES(2560, 1)), "copies": (torch.bfloat16, [0, 100, 2560])}[name]
    tj, tk = ES(4096, 1), ES(2048, 1)
    a, b, c = ja.Relation([2560, 4096], [ti, tj], dt), ja.Relation([4096, 2048], [tj, tk], dt), ja.Relation([2560, 2048], [ti, tk], dt)
    before = ja.ja_launch_count()
    ja.Spec("ij,jk->ik", {"i": ti, "j": tj, "k": tk}).execute([a, b], c)
    torch.cuda.synchronize()
    print(ja.ja_launch_count() - before)
"""


# 80 tiles over 74 pairs of SMs: a launch of whole tiles and one of split ones, whichever product the process plans first
@pytest.mark.parametrize("order", [("f16", "bf16"), ("bf16", "f16"), ("copies", "f16", "bf16")])
def test_split_whatever_was_planned_first(order):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", FIRST_PLANS, *order], cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    assert out.stdout.split() == ["3" if name == "copies" else "2" for name in order]

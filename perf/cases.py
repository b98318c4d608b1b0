"""The measured work of this library: what a program that uses it has it do, one call or one chain of calls at a time.

Every case goes through the public entry points of paper_2609_03905_b200 (`Spec.execute`, `Spec.execute_join`,
`repartition`, `repartition_agg`, `from_dense`, `to_dense`, `LlamaBlock.forward`) on relations that the program holds on
the GPU. `listed()` names twelve of them; `draw()` gives further ones of the same kinds, with the sizes, tilings, cell
types and options spread over the range each kind is used in, sizes that are no multiple of any tile among them.

Interval counts (`gi`, `gj`, ...) cut an index into near-equal intervals, as `equal_splits` does.
"""
import math

import torch

import paper_2609_03905_b200 as ja
from paper_2609_03905_b200.llama_block import LlamaBlock

ES = ja.equal_splits
DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
HEAD_DIM = 128   # the attention operator's last index


def listed():
    return [
        # one small matmul join-agg, 64 x 64 sub-tensors: what a call costs when there is next to no arithmetic in it
        {"name": "matmul_f32_256", "kind": "matmul", "dtype": "f32", "m": 256, "k": 256, "n": 256, "gi": 4, "gj": 4, "gk": 4},
        # a projection of few tokens (a decoding step's batch): the weights are read once and used 32 times
        {"name": "projection_32_tokens", "kind": "matmul", "dtype": "bf16", "m": 32, "k": 4096, "n": 11008, "gi": 1, "gj": 8, "gk": 8},
        # a plan that cuts only the contracted index, 64 ways: 172-cell block rows, as the optimizer may return for 64 function specs
        {"name": "contraction_cut_64", "kind": "matmul", "dtype": "bf16", "m": 2048, "k": 11008, "n": 4096, "gi": 1, "gj": 64, "gk": 1},
        # the SwiGLU MLP of 2048 tokens as four chained join-aggs, every index cut eight ways (1376-wide FFN blocks)
        {"name": "mlp_2048_tokens", "kind": "mlp", "dtype": "bf16", "tokens": 2048, "hidden": 4096, "ffn": 11008, "gi": 8, "gj": 8, "gk": 8},
        # causal attention at the 7B shape, 128-row blocks
        {"name": "attention_b4_s2048", "kind": "attention", "dtype": "bf16", "batch": 4, "seq": 2048, "heads": 32, "kv_heads": 32, "ends": "",
         "cut": 128, "causal": True, "lse": False},
        # grouped-query attention over sequences packed one after the other, of the lengths prompts have: no multiple of any tile
        {"name": "attention_packed_gqa", "kind": "attention", "dtype": "f16", "batch": 1, "seq": 6001, "heads": 32, "kv_heads": 8,
         "ends": "777,1291,3000,4633,6001", "cut": 0, "causal": True, "lse": False},
        # softmax of the scores of 32 heads, 256-column blocks, as one join-agg
        {"name": "softmax_32x2048x2048", "kind": "rows", "op": "softmax", "fused": True, "dtype": "bf16", "outer": 32, "rows": 2048,
         "width": 2048, "gi": 8, "gj": 8},
        # an activation re-tiled from eight column blocks to one head per block, between two operators of a plan
        {"name": "relayout_16384x4096", "kind": "relayout", "op": "repartition", "dtype": "bf16", "rows": 16384, "cols": 4096, "src_i": 128, "src_j": 8,
         "dst_i": 128, "dst_j": 32},
        # a producer executed through its join, the contracted index cut four ways, and the aggregating relayout its consumer runs
        {"name": "join_then_aggregate", "kind": "aggregate", "dtype": "bf16", "partial": "f32", "m": 4096, "k": 11008, "n": 4096, "gi": 4, "gj": 4,
         "gk": 8, "dst_i": 32, "dst_k": 8},
        # a contraction outside the two-index form: scores of 32 heads as a batched product
        {"name": "einsum_batched_scores", "kind": "einsum", "einsum": "bij,bkj->bik", "fn": "mul", "agg": "sum", "dtype": "bf16", "out": "bf16",
         "b": 32, "i": 512, "j": 128, "k": 512, "cut": 4},
        # the paper's block on one sequence of 1024 tokens in its precision: many launches of tens of microseconds
        {"name": "block_gqa_1x1024", "kind": "block", "dtype": "f16", "batch": 1, "seq": 1024, "hidden": 4096, "kv_heads": 8, "ffn": 14336,
         "token_block": 128, "plan": "mixed"},
        # the 7B block on 8 x 2048 tokens: the throughput case
        {"name": "block_7b_8x2048", "kind": "block", "dtype": "bf16", "batch": 8, "seq": 2048, "hidden": 4096, "kv_heads": 32, "ffn": 11008,
         "token_block": 128, "plan": "mixed"},
    ]


# ---- further cases of the same ranges ---------------------------------------------------------------------------
def _size(rng, lo, hi, odd=0.5):
    """An extent spread over the logarithm of [lo, hi]; with probability `odd` any number, else a multiple of 64."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, n) if rng.random() < odd or n < 64 else max(64, n // 64 * 64)


def _draw_matmul(rng):
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    m, k, n = _size(rng, 8, 16384), _size(rng, 256, 11008), _size(rng, 256, 11008)
    if dtype == "f32":   # the type of small and of exact problems
        m, k, n = _size(rng, 64, 2048), _size(rng, 64, 4096), _size(rng, 64, 4096)
    cuts = [1, 2, 4, 8]
    return {"kind": "matmul", "dtype": dtype, "m": m, "k": k, "n": n, "gi": rng.choice([g for g in cuts if g * 8 <= m]), "gj": rng.choice(cuts),
            "gk": rng.choice(cuts)}


def _draw_mlp(rng):
    hidden = rng.choice([512, 1024, 2048, 4096])
    ffn = rng.choice([hidden * 43 // 16, hidden * 7 // 2])     # the 7B and the paper's ratio
    return {"kind": "mlp", "dtype": rng.choice(["bf16", "f16"]), "tokens": _size(rng, 32, 8192), "hidden": hidden, "ffn": ffn,
            "gi": rng.choice([1, 2, 4]), "gj": rng.choice([1, 4, 8]), "gk": rng.choice([1, 4, 8])}


def _draw_attention(rng):
    seq, cut = _size(rng, 64, 8192, odd=0.0) // 64 * 64, 64
    if seq % 128 == 0:
        cut = 128
    ends = ""
    if rng.random() < 0.5:   # lengths as they come
        seq, cut = _size(rng, 65, 8192, odd=1.0), 0
    if rng.random() < 0.4 and seq >= 512:
        step = cut or 1
        inner = sorted({rng.randrange(step, seq, step) for _ in range(rng.choice([1, 3, 5]))})
        ends = ",".join(str(e) for e in inner + [seq])
    heads = rng.choice([4, 8, 16, 32])
    batch = rng.choice([b for b in (1, 2, 3, 4, 8) if b * seq <= 16384])
    return {"kind": "attention", "dtype": rng.choice(["bf16", "f16"]), "batch": batch, "seq": seq, "heads": heads,
            "kv_heads": heads // rng.choice([1, 1, 4]), "ends": ends, "cut": cut, "causal": rng.random() < 0.75, "lse": rng.random() < 0.25}


def _draw_rows(rng):
    op = rng.choice(["rmsnorm", "softmax"])
    width = _size(rng, 128, 16384)
    outer = rng.choice([1, 4, 32]) if op == "softmax" else 1
    rows = _size(rng, 16, max(16, min(16384, (1 << 26) // (width * outer))))
    return {"kind": "rows", "op": op, "fused": rng.random() < 0.6, "dtype": rng.choice(["bf16", "bf16", "f16", "f32"]), "outer": outer, "rows": rows,
            "width": width, "gi": rng.choice([1, 2, 8]), "gj": rng.choice([1, 4, 8])}


def _draw_relayout(rng):
    rows, cols = _size(rng, 64, 32768), _size(rng, 64, 8192)
    cuts_i, cuts_j = [g for g in (1, 4, 16, 64, 128) if g <= rows], [1, 2, 8, 32]
    return {"kind": "relayout", "op": rng.choice(["repartition", "repartition", "pack"]), "dtype": rng.choice(["bf16", "bf16", "f16", "f32"]),
            "rows": rows, "cols": cols, "src_i": rng.choice(cuts_i), "src_j": rng.choice(cuts_j), "dst_i": rng.choice(cuts_i),
            "dst_j": rng.choice(cuts_j)}


def _draw_aggregate(rng):
    dtype = rng.choice(["bf16", "bf16", "f16"])
    gi, gj = rng.choice([1, 2, 4]), rng.choice([2, 4, 8])
    # function specs of one shape: every index a multiple of its interval count
    m, k, n = (_size(rng, 256, 8192) // gi * gi, _size(rng, 512, 11008, odd=0.0) // (gj * 8) * gj * 8, _size(rng, 256, 4096, odd=0.25) // 64 * 64)
    return {"kind": "aggregate", "dtype": dtype, "partial": rng.choice([dtype, "f32"]), "m": m, "k": k, "n": n, "gi": gi, "gj": gj,
            "gk": rng.choice([1, 2, 4]), "dst_i": rng.choice([1, 8]), "dst_k": rng.choice([1, 4, 8])}


_EINSUMS = [("bij,bjk->bik", "mul", "sum"), ("bij,bkj->bik", "mul", "sum"), ("ij,kj->ik", "mul", "sum"), ("ji,jk->ik", "mul", "sum"),
            ("ij,j->i", "mul", "sum"), ("bij->bj", "ident", "max"), ("bij->b", "square", "sum"), ("i,k->ik", "mul", "none")]


def _draw_einsum(rng):
    einsum, fn, agg = rng.choice(_EINSUMS)
    dtype = rng.choice(["bf16", "f16", "f32"])
    return {"kind": "einsum", "einsum": einsum, "fn": fn, "agg": agg, "dtype": dtype, "out": "f32" if fn == "square" else rng.choice([dtype, "f32"]),
            "b": _size(rng, 2, 32), "i": _size(rng, 32, 512), "j": _size(rng, 32, 512), "k": _size(rng, 32, 512), "cut": rng.choice([1, 2, 4])}


def _draw_block(rng):
    hidden = rng.choice([512, 1024, 2048, 4096])
    heads = hidden // HEAD_DIM
    token_block = rng.choice([128, 128, 64, 200, 125])
    seq = token_block * rng.choice([1, 2, 3, 4, 8])
    batch = rng.choice([b for b in (1, 2, 3, 5, 8, 16) if b * seq <= 8192])
    return {"kind": "block", "dtype": rng.choice(["bf16", "f16"]), "batch": batch, "seq": seq, "hidden": hidden,
            "kv_heads": rng.choice([heads, heads // 4]), "ffn": rng.choice([hidden * 43 // 16, hidden * 7 // 2]), "token_block": token_block,
            "plan": rng.choice(["mixed", "mixed", "seq", "head"])}


def draw(rng):
    return rng.choice([_draw_matmul, _draw_matmul, _draw_mlp, _draw_attention, _draw_attention, _draw_rows, _draw_relayout, _draw_aggregate,
                       _draw_einsum, _draw_block])(rng)


# ---- what the program has in hand ---------------------------------------------------------------------------------
def _normal(gen, shape, dtype, std=1.0, mean=0.0):
    return torch.randn(list(shape), generator=gen, device="cuda", dtype=torch.float32).mul_(std).add_(mean).to(dtype)


def _relation(gen, shape, splits, dtype, std=1.0, mean=0.0):
    return ja.from_dense(_normal(gen, shape, dtype, std, mean), splits)


def _prepare_matmul(c, gen):
    dt = DTYPES[c["dtype"]]
    ti, tj, tk = ES(c["m"], c["gi"]), ES(c["k"], c["gj"]), ES(c["n"], c["gk"])
    a = _relation(gen, (c["m"], c["k"]), [ti, tj], dt)
    b = _relation(gen, (c["k"], c["n"]), [tj, tk], dt, 0.02)
    return {"a": a, "b": b, "c": ja.Relation([c["m"], c["n"]], [ti, tk], dt), "spec": ja.Spec("ij,jk->ik", {"i": ti, "j": tj, "k": tk})}


def _run_matmul(s):
    s["spec"].execute([s["a"], s["b"]], s["c"])
    return s["c"].payload


def _prepare_mlp(c, gen):
    dt, t, d, f = DTYPES[c["dtype"]], c["tokens"], c["hidden"], c["ffn"]
    ti, td, tf = ES(t, c["gi"]), ES(d, c["gj"]), ES(f, c["gk"])
    s = {"x": _relation(gen, (t, d), [ti, td], dt), "w1": _relation(gen, (d, f), [td, tf], dt, 0.02),
         "w3": _relation(gen, (d, f), [td, tf], dt, 0.02), "w2": _relation(gen, (f, d), [tf, td], dt, 0.02)}
    s.update({n: ja.Relation([t, f], [ti, tf], dt) for n in "abh"}, y=ja.Relation([t, d], [ti, td], dt))
    s["up"] = ja.Spec("ij,jk->ik", {"i": ti, "j": td, "k": tf})
    s["gate"] = ja.Spec("ij,ij->ij", {"i": ti, "j": tf}, "silu_mul", (), "none")
    s["down"] = ja.Spec("ij,jk->ik", {"i": ti, "j": tf, "k": td})
    return s


def _run_mlp(s):
    s["up"].execute([s["x"], s["w1"]], s["a"])
    s["up"].execute([s["x"], s["w3"]], s["b"])
    s["gate"].execute([s["a"], s["b"]], s["h"])
    s["down"].execute([s["h"], s["w2"]], s["y"])
    return {"h": s["h"].payload, "y": s["y"].payload}


def _ends(c):
    return [int(e) for e in c["ends"].split(",")] if c["ends"] else []


def _prepare_attention(c, gen):
    dt, b, n, h, g = DTYPES[c["dtype"]], c["batch"], c["seq"], c["heads"], c["kv_heads"]
    ends = _ends(c)
    # rows: blocks of `cut` positions, or one block per sequence
    tq = ES(n, n // c["cut"]) if c["cut"] else [0] + (ends or [n])
    tg = ES(g, g)
    th = [v * (h // g) for v in tg]
    q_sp, k_sp = [ES(b, b), tq, th, [0, HEAD_DIM]], [ES(b, b), tq, tg, [0, HEAD_DIM]]
    s = {"q": _relation(gen, (b, n, h, HEAD_DIM), q_sp, dt), "k": _relation(gen, (b, n, g, HEAD_DIM), k_sp, dt),
         "v": _relation(gen, (b, n, g, HEAD_DIM), k_sp, dt), "o": ja.Relation([b, n, h, HEAD_DIM], q_sp, dt)}
    s["lse"] = ja.Relation([b, n, h], q_sp[:3], torch.float32) if c["lse"] else None
    params = (1.0 / math.sqrt(HEAD_DIM), 1.0 if c["causal"] else 0.0) + tuple(float(e) for e in ends)
    parts = {"b": q_sp[0], "q": tq, "h": th, "d": [0, HEAD_DIM], "k": tq}
    if g == h:
        s["spec"] = ja.Spec("bqhd,bkhd,bkhd->bqhd", parts, "attention", params, "online_softmax")
    else:
        s["spec"] = ja.Spec("bqhd,bkgd,bkgd->bqhd", dict(parts, g=tg), "attention", params, "online_softmax")
    return s


def _run_attention(s):
    if s["lse"] is None:
        s["spec"].execute([s["q"], s["k"], s["v"]], s["o"])
        return s["o"].payload
    s["spec"].execute([s["q"], s["k"], s["v"]], [s["o"], s["lse"]])
    return {"o": s["o"].payload, "lse": s["lse"].payload}


def _prepare_rows(c, gen):
    dt, r, w = DTYPES[c["dtype"]], c["rows"], c["width"]
    ti, tj = ES(r, min(c["gi"], r)), ES(w, c["gj"])
    s = {"op": c["op"], "fused": c["fused"]}
    if c["op"] == "rmsnorm":
        parts, eps = {"i": ti, "j": tj}, (1e-5,)
        s.update(x=_relation(gen, (r, w), [ti, tj], dt, 2.0), g=_relation(gen, (w,), [tj], dt, 0.1, 1.0), y=ja.Relation([r, w], [ti, tj], dt),
                 stat=ja.Relation([r], [ti], torch.float32))
        s["norm"] = ja.Spec("ij,j->ij", parts, "rmsnorm", eps, "none")
        s["sumsq"] = ja.Spec("ij->i", parts, "square", (), "sum")
        s["scale"] = ja.Spec("ij,i,j->ij", parts, "rms_scale", eps, "none")
    else:
        th = ES(c["outer"], c["outer"])
        parts, sp = {"h": th, "i": ti, "j": tj}, [th, ti, tj]
        s.update(x=_relation(gen, (c["outer"], r, w), sp, dt, 2.0), y=ja.Relation([c["outer"], r, w], sp, dt),
                 stat=ja.Relation([c["outer"], r], sp[:2], torch.float32), den=ja.Relation([c["outer"], r], sp[:2], torch.float32))
        s["norm"] = ja.Spec("hij->hij", parts, "softmax", (), "none")
        s["max"] = ja.Spec("hij->hi", parts, "ident", (), "max")
        s["expsum"] = ja.Spec("hij,hi->hi", parts, "exp_sub", (), "sum")
        s["divide"] = ja.Spec("hij,hi,hi->hij", parts, "exp_sub_div", (), "none")
    return s


def _run_rows(s):
    if s["op"] == "rmsnorm":
        if s["fused"]:
            s["norm"].execute([s["x"], s["g"]], s["y"])
            return s["y"].payload
        s["sumsq"].execute([s["x"]], s["stat"])
        s["scale"].execute([s["x"], s["stat"], s["g"]], s["y"])
        return {"y": s["y"].payload, "stat": s["stat"].payload}
    if s["fused"]:
        s["norm"].execute([s["x"]], s["y"])
        return s["y"].payload
    s["max"].execute([s["x"]], s["stat"])
    s["expsum"].execute([s["x"], s["stat"]], s["den"])
    s["divide"].execute([s["x"], s["stat"], s["den"]], s["y"])
    return {"y": s["y"].payload, "stat": s["stat"].payload, "den": s["den"].payload}


def _prepare_relayout(c, gen):
    dt, shape = DTYPES[c["dtype"]], [c["rows"], c["cols"]]
    src, dst = [ES(c["rows"], c["src_i"]), ES(c["cols"], c["src_j"])], [ES(c["rows"], c["dst_i"]), ES(c["cols"], c["dst_j"])]
    if c["op"] == "pack":   # a dense tensor becomes a relation and the relation a dense tensor again
        return {"op": "pack", "dense": _normal(gen, shape, dt), "splits": dst}
    return {"op": "repartition", "src": _relation(gen, shape, src, dt), "dst": ja.Relation(shape, dst, dt)}


def _run_relayout(s):
    if s["op"] == "pack":
        rel = ja.from_dense(s["dense"], s["splits"])
        return {"relation": rel.payload, "dense": ja.to_dense(rel)}
    ja.repartition(s["src"], s["dst"])
    return s["dst"].payload


def _prepare_aggregate(c, gen):
    dt, pdt = DTYPES[c["dtype"]], DTYPES[c["partial"]]
    ti, tj, tk = ES(c["m"], c["gi"]), ES(c["k"], c["gj"]), ES(c["n"], c["gk"])
    return {"a": _relation(gen, (c["m"], c["k"]), [ti, tj], dt), "b": _relation(gen, (c["k"], c["n"]), [tj, tk], dt, 0.02),
            "p": ja.partial_relation(c["gj"], [c["m"], c["n"]], [ti, tk], pdt),
            "y": ja.Relation([c["m"], c["n"]], [ES(c["m"], c["dst_i"]), ES(c["n"], c["dst_k"])], dt),
            "spec": ja.Spec("ij,jk->ik", {"i": ti, "j": tj, "k": tk})}


def _run_aggregate(s):
    s["spec"].execute_join([s["a"], s["b"]], s["p"])
    ja.repartition_agg(s["p"], "sum", s["y"])
    return {"partials": s["p"].payload, "y": s["y"].payload}


def _terms(c):
    ins, out = c["einsum"].split("->")
    return ins.split(","), out


def _prepare_einsum(c, gen):
    ins, out = _terms(c)
    cuts = {x: ES(c[x], min(c["cut"], c[x])) for x in "bijk"}
    # operands after the first are scaled so that products of long sums stay of order one
    rels = [_relation(gen, [c[x] for x in t], [cuts[x] for x in t], DTYPES[c["dtype"]], 1.0 if n == 0 else 0.1) for n, t in enumerate(ins)]
    letters = sorted(set("".join(ins)))
    return {"ins": rels, "out": ja.Relation([c[x] for x in out], [cuts[x] for x in out], DTYPES[c["out"]]),
            "spec": ja.Spec(c["einsum"], {x: cuts[x] for x in letters}, c["fn"], (), c["agg"])}


def _run_einsum(s):
    s["spec"].execute(s["ins"], s["out"])
    return s["out"].payload


def _prepare_block(c, gen):
    dt, d, f = DTYPES[c["dtype"]], c["hidden"], c["ffn"]
    kv = c["kv_heads"] * HEAD_DIM
    shapes = {"wq": (d, d), "wk": (d, kv), "wv": (d, kv), "wo": (d, d), "w1": (d, f), "w3": (d, f), "w2": (f, d)}
    w = {n: _normal(gen, sh, dt, 0.02) for n, sh in shapes.items()}
    w.update({n: _normal(gen, (d,), dt, 0.1, 1.0) for n in ("g1", "g2")})
    heads = d // HEAD_DIM
    blk = LlamaBlock(c["batch"], c["seq"], d, heads, f, w, plan=c["plan"], token_block=c["token_block"], col_blocks=min(8, heads),
                     n_kv_heads=c["kv_heads"], dtype=dt)
    x = ja.from_dense(_normal(gen, (c["batch"] * c["seq"], d), dt), [blk.t_sp, blk.io_c])
    ja.repartition(x, blk.x)
    torch.cuda.current_stream().synchronize()
    return {"block": blk}


def _run_block(s):
    blk = s["block"]
    out = blk.forward()
    return {"out": out.payload, "k": blk.ka.payload, "v": blk.va.payload}   # the layer's output and what a cache would keep


_KINDS = {"matmul": (_prepare_matmul, _run_matmul), "mlp": (_prepare_mlp, _run_mlp), "attention": (_prepare_attention, _run_attention),
          "rows": (_prepare_rows, _run_rows), "relayout": (_prepare_relayout, _run_relayout), "aggregate": (_prepare_aggregate, _run_aggregate),
          "einsum": (_prepare_einsum, _run_einsum), "block": (_prepare_block, _run_block)}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    state = _KINDS[case["kind"]][0](case, gen)
    state["run"] = _KINDS[case["kind"]][1]
    return state


def run(state):
    return state["run"](state)


# ---- what one pass cannot do without ---------------------------------------------------------------------------------
def _esize(name):
    return DTYPES[name].itemsize


def work(case):
    c, kind = case, case["kind"]
    e = _esize(c["dtype"])
    if kind == "matmul":
        return {"bytes": e * (c["m"] * c["k"] + c["k"] * c["n"] + c["m"] * c["n"]), "flops": 2.0 * c["m"] * c["k"] * c["n"]}
    if kind == "mlp":   # h is returned: written once beside y
        t, d, f = c["tokens"], c["hidden"], c["ffn"]
        return {"bytes": e * (2 * t * d + t * f + 3 * d * f), "flops": 6.0 * t * d * f}
    if kind == "attention":
        b, n, h, g = c["batch"], c["seq"], c["heads"], c["kv_heads"]
        ends = _ends(c) or [n]
        pairs = sum(l * (l + 1) / 2 if c["causal"] else l * l for l in (y - x for x, y in zip([0] + ends, ends)))
        return {"bytes": e * HEAD_DIM * b * n * (2 * h + 2 * g) + (4 * b * n * h if c["lse"] else 0), "flops": 4.0 * b * h * HEAD_DIM * pairs}
    if kind == "rows":
        cells = c["outer"] * c["rows"] * c["width"]
        passes = 2 if c["fused"] else 3 if c["op"] == "rmsnorm" else 4   # separate join-aggs read their input each on its own
        return {"bytes": e * cells * passes, "flops": 0.0}
    if kind == "relayout":
        return {"bytes": e * c["rows"] * c["cols"] * (4 if c["op"] == "pack" else 2), "flops": 0.0}
    if kind == "aggregate":   # the partial relation is an output of the first call and the input of the second
        mn = c["m"] * c["n"]
        return {"bytes": e * (c["m"] * c["k"] + c["k"] * c["n"] + mn) + 2 * c["gj"] * mn * _esize(c["partial"]), "flops": 2.0 * c["k"] * mn}
    if kind == "einsum":
        ins, out = _terms(c)
        size = lambda t: math.prod(c[x] for x in t)   # noqa: E731
        return {"bytes": e * sum(size(t) for t in ins) + _esize(c["out"]) * size(out),
                "flops": 2.0 * size(sorted(set("".join(ins)))) if len(ins) > 1 else 0.0}
    t, d, f, kv = c["batch"] * c["seq"], c["hidden"], c["ffn"], c["kv_heads"] * HEAD_DIM
    return {"bytes": e * (2 * d * d + 2 * d * kv + 3 * d * f + 2 * t * d + 2 * t * kv),
            "flops": 2.0 * t * d * (2 * d + 2 * kv) + 6.0 * t * d * f + 2.0 * t * c["seq"] * d}


def tolerance(case):
    """Relayouts move bits. Everything else accumulates in f32 and rounds once per stored cell: half an ulp of the cell type
    (2^-9 bf16, 2^-12 f16) per rounding, a few roundings along a chain; f32 results differ by the order of their sums."""
    if case["kind"] == "relayout" or (case["kind"] == "einsum" and case["agg"] == "max"):
        return "exact"
    return {"f32": {"rel": 1e-5, "max": 2e-4}, "f16": {"rel": 1.5e-3, "max": 3e-2}, "bf16": {"rel": 1e-2, "max": 0.2}}[case["dtype"]]

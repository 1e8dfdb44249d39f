"""What a program that serves or builds a Tetra model has this library do, as cases that can be timed and compared.

A case is a dict of plain values; "kind" says which public entry points it goes through:

  gemv     one matrix, one activation vector: tetra_gemv (zero-pad rule) or tetra_gemv_tail (tail rule)
  list     the independent matrices of one dependency step of a layer: tetra_gemv_list
  layer    a whole layer in model order, four dependent steps: four tetra_gemv_list calls
  pass     all projections of several layers as one planned list: tetra_gemv_grouped_run
  batched  one matrix, several activation vectors: tetra_gemv_batched
  q4       a 4-bit matrix (output head, int4 projection): tetra_q4_gemv
  q4list   the int4 projections of several layers as one planned list: tetra_q4_list_run
  q4rows   embedding rows of a prompt's tokens: tetra_q4_rows
  encode   the encoder's search: tetra_encode_blocks
  load     a layer brought into the kernels' layouts and checked: tetra_pack_codes + tetra_decode_packed for the
           Tetra matrices, tetra_q4_pack + tetra_q4_rows for the int4 ones

Shapes are those of shapes.py (three dense models, two single-matrix configurations) and generic sizes around
them.  Codes are uniform 48-bit words (every word is legal), row scales exp(-4 + 0.3 z), activations float16
N(0, 1), tails row scale times N(0, 1); 4-bit matrices have uniform nibbles, scales exp(-5 + 0.3 z) and offsets
that centre a group on zero; encoder blocks are Gaussian weights at their row's scale.
"""
import math

import torch

from paper_2609_35465_b200 import shapes, tetra

DEVICE = "cuda"


def listed():
    return [
        # the smallest product a model has: one square-ish projection, one token; latency is all there is
        dict(name="gemv_2048x2304", kind="gemv", N=2048, K=2304, rule="tail"),
        # odd rows, odd inputs, K not a multiple of 24 or 8: zero-pad rule, nothing aligned
        dict(name="gemv_ragged_5003x7001", kind="gemv", N=5003, K=7001, rule="pad"),
        # q, k and v of an 8B layer: one step of a decode loop
        dict(name="list_qkv_8b", kind="list", rows="4096,1024,1024", K=4096),
        # a 4B layer the way a decode loop runs it: q,k,v | o | gate,up | down
        dict(name="layer_4b", kind="layer", hidden=2560, inter=9728, q=4096, kv=1024),
        # every projection of the 8B model for one token, planned once
        dict(name="pass_8b", kind="pass", hidden=4096, inter=12288, q=4096, kv=1024, layers=36),
        # a few sequences decoded together, an odd number of them
        dict(name="batched_3_4096x4096", kind="batched", N=4096, K=4096, batch=3),
        # as many sequences as the call takes, the largest projection
        dict(name="batched_16_4096x12288", kind="batched", N=4096, K=12288, batch=16),
        # logits of one token: the head over the whole vocabulary
        dict(name="q4_head_151936x4096", kind="q4", N=151936, K=4096, G=64, batch=1),
        # the v, o and down projections of the 8B model as int4, one token, planned once
        dict(name="q4list_8b", kind="q4list", hidden=4096, inter=12288, q=4096, kv=1024, layers=36),
        # the token embeddings of a prompt
        dict(name="q4rows_1024x4096", kind="q4rows", N=151936, K=4096, count=1024),
        # a slice of a matrix through the encoder
        dict(name="encode_24576", kind="encode", blocks=24576),
        # one 8B layer read from a file into the kernels' layouts, and checked
        dict(name="load_layer_8b", kind="load", hidden=4096, inter=12288, q=4096, kv=1024),
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], its logarithm uniform."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gemv", "gemv", "list", "layer", "pass", "batched", "batched", "q4", "q4", "q4list", "q4rows",
                       "encode", "load"])
    if kind == "gemv":
        return dict(kind=kind, N=_spread(rng, 512, 17408), K=_spread(rng, 768, 17408), rule=rng.choice(["tail", "pad"]))
    if kind == "list":
        rows = [_spread(rng, 256, 12288) for _ in range(rng.randint(2, 8))]
        return dict(kind=kind, rows=",".join(str(r) for r in rows), K=_spread(rng, 1024, 8192))
    if kind in ("layer", "pass", "q4list", "load"):
        hidden = 128 * _spread(rng, 8, 40)                    # 1024 .. 5120
        kv = 128 * rng.choice([2, 4, 8])
        case = dict(kind=kind, hidden=hidden, inter=128 * _spread(rng, hidden // 64, hidden * 27 // 1000 + hidden // 1280),
                    q=128 * rng.choice([16, 32, 40]), kv=kv)
        if kind == "load":
            case["inter"] = min(case["inter"], 12288)
            case["hidden"] = min(case["hidden"], 4096)
        if kind in ("pass", "q4list"):
            layer = sum(n * k for n, k in _layer_shapes(case))
            full = sum(n * k for n, k in _layer_shapes(dict(hidden=4096, inter=12288, q=4096, kv=1024))) * 36
            case["layers"] = _spread(rng, 1, max(1, min(40, full // layer)))
        return case
    if kind == "batched":
        K = _spread(rng, 768, 12288)
        return dict(kind=kind, N=_spread(rng, 512, 12288), K=rng.choice([K, K - K % 24]), batch=rng.randint(2, 16))
    if kind == "q4":
        G = rng.choice([64, 128])
        return dict(kind=kind, N=_spread(rng, 1000, 151936), K=G * _spread(rng, 1024 // G, 4096 // G), G=G,
                    batch=rng.choice([1, 1, 2, 3, 4, 5, 8]))
    if kind == "q4rows":
        return dict(kind=kind, N=_spread(rng, 32000, 151936), K=64 * _spread(rng, 16, 64), count=_spread(rng, 1, 4096))
    return dict(kind=kind, blocks=_spread(rng, 100, 24576))


# ---------------------------------------------------------------------------
# shapes
# ---------------------------------------------------------------------------
def _model(case):
    return shapes.Model("case", case.get("layers", 1), case["hidden"], case["inter"], case["q"] // 128, case["kv"] // 128)


def _layer_shapes(case):
    return [(m.N, m.K) for m in _model(case).layer_matrices()]


def _int4_shapes(case):
    """v, o and down of a layer, where the 4-bit groups of 128 fit."""
    return [(m.N, m.K) for m in _model(case).layer_matrices() if m.name in ("v", "o", "down")]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _bytes(g, n):
    """n random bytes on the device."""
    return torch.randint(-(1 << 62), 1 << 62, (-(-n // 4),), dtype=torch.int64, device=DEVICE, generator=g).to(
        torch.int32).view(torch.uint8)[:n]


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float32, device=DEVICE, generator=g)


def _table():
    return tetra.tetra_build_table((4.3156, 5.4415), device=DEVICE)


def _matrix(g, table, N, K, rule, x, y):
    """A Tetra matrix in the kernels' layout, with the vectors it reads and writes."""
    tail_rule = rule == "tail"
    B = K // 24 if tail_rule else -(-K // 24)
    packed = tetra.tetra_pack_codes(_bytes(g, 6 * N * B).reshape(N, B, 6), table, N, B)
    sigma = torch.exp(-4.0 + 0.3 * _normal(g, N))
    tail = None
    if tail_rule and K % 24:
        tail = (sigma[:, None] * _normal(g, N, K % 24)).to(torch.float16)
    return dict(codes=packed, row_scales=sigma, x=x, tail=tail, y=y, N=N, K=K)


def _vectors(g, batch, K):
    return _normal(g, batch, K).to(torch.float16)


def _q4_source(g, N, K, G):
    """A 4-bit matrix in file order: nibbles, scales, offsets."""
    q = _bytes(g, N * (K // 2)).reshape(N, K // 2)
    scale = torch.exp(-5.0 + 0.3 * _normal(g, N, K // G)).to(torch.float16)
    offset = (-scale.float() * (7.5 + 0.5 * _normal(g, N, K // G))).to(torch.float16)
    return q, scale, offset


def _zeros(*shape):
    return torch.zeros(*shape, dtype=torch.float32, device=DEVICE)


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed)
    s = dict(kind=kind)
    if kind in ("gemv", "list", "layer", "pass", "batched", "encode", "load"):
        s["table"] = _table()
    if kind == "gemv":
        N, K = case["N"], case["K"]
        s["rule"] = case["rule"]
        s["m"] = _matrix(g, s["table"], N, K, case["rule"], _vectors(g, 1, K)[0], _zeros(N))
    elif kind == "list":
        K = case["K"]
        x = _vectors(g, 1, K)[0]                      # the matrices of a step read the same activations
        s["items"] = [_matrix(g, s["table"], int(n), K, "tail", x, _zeros(int(n))) for n in case["rows"].split(",")]
        s["problems"] = tetra.make_problems(s["items"])
    elif kind == "layer":
        items = [_matrix(g, s["table"], n, k, "tail", None, _zeros(n)) for n, k in _layer_shapes(case)]
        xs = [_vectors(g, 1, k)[0] for k in (case["hidden"], case["q"], case["hidden"], case["inter"])]
        for it, step in zip(items, (0, 0, 0, 1, 2, 2, 3)):
            it["x"] = xs[step]
        s["items"] = items
        s["steps"] = [tetra.make_problems(items[a:b]) for a, b in ((0, 3), (3, 4), (4, 6), (6, 7))]
    elif kind == "pass":
        mats = _layer_shapes(case) * case["layers"]
        s["y"] = _zeros(sum(-(-n // 4) * 4 for n, _ in mats))
        s["x"] = torch.zeros(sum(-(-k // 8) * 8 for _, k in mats), dtype=torch.float16, device=DEVICE)
        s["x"].copy_(_normal(g, s["x"].numel()))
        items, xo, yo = [], 0, 0
        for n, k in mats:
            items.append(_matrix(g, s["table"], n, k, "tail", s["x"][xo:xo + k], s["y"][yo:yo + n]))
            xo += -(-k // 8) * 8
            yo += -(-n // 4) * 4
        s["items"] = items
        problems = tetra.make_problems(items)
        s["ws"] = torch.empty(tetra.tetra_grouped_workspace_bytes(problems), dtype=torch.uint8, device=DEVICE)
        tetra.tetra_gemv_grouped_plan(problems, s["ws"])
    elif kind == "batched":
        N, K, V = case["N"], case["K"], case["batch"]
        s["m"] = _matrix(g, s["table"], N, K, "tail", _vectors(g, V, K), _zeros(V, N))
        s["batch"] = V
        s["ws"] = torch.empty(tetra.tetra_batched_workspace_bytes(N, K), dtype=torch.uint8, device=DEVICE)
    elif kind == "q4":
        N, K, G, V = case["N"], case["K"], case["G"], case["batch"]
        s.update(N=N, K=K, G=G, batch=V, x=_vectors(g, V, K), y=_zeros(V, N))
        s["packed"] = tetra.tetra_q4_pack(*_q4_source(g, N, K, G), N, K, G)
    elif kind == "q4list":
        mats = _int4_shapes(case) * case["layers"]
        s["y"] = _zeros(sum(n for n, _ in mats))
        items, yo = [], 0
        for n, k in mats:
            items.append(dict(packed=tetra.tetra_q4_pack(*_q4_source(g, n, k, 128), n, k, 128), x=_vectors(g, 1, k)[0],
                              y=s["y"][yo:yo + n], N=n, K=k))
            yo += n
        s["items"] = items
        s["ws"] = tetra.tetra_q4_list_plan(tetra.make_q4_problems(items), 128)
    elif kind == "q4rows":
        N, K, n = case["N"], case["K"], case["count"]
        s.update(N=N, K=K, packed=tetra.tetra_q4_pack(*_q4_source(g, N, K, 64), N, K, 64))
        s["ids"] = torch.randint(0, N, (n,), dtype=torch.int32, device=DEVICE, generator=g)
        s["out"] = torch.empty((n, K), dtype=torch.float16, device=DEVICE)
    elif kind == "encode":
        n = case["blocks"]
        s["sigma"] = torch.exp(-4.0 + 0.3 * _normal(g, n))
        s["w"] = s["sigma"][:, None] * _normal(g, n, 24)
    elif kind == "load":
        s["tetra"], s["q4"] = [], []
        int4 = _int4_shapes(case)
        for n, k in _layer_shapes(case)[:2] + _layer_shapes(case)[4:6]:      # q, k, gate, up
            s["tetra"].append((n, k // 24, _bytes(g, 6 * n * (k // 24)).reshape(n, k // 24, 6)))
        for n, k in int4:                                                    # v, o, down
            s["q4"].append((n, k, _q4_source(g, n, k, 128),
                            torch.randint(0, n, (64,), dtype=torch.int32, device=DEVICE, generator=g)))
    else:
        raise ValueError(kind)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "gemv":
        m = s["m"]
        if s["rule"] == "tail":
            return tetra.tetra_gemv_tail(m["codes"], m["row_scales"], s["table"], m["x"], m["y"], m["N"], m["K"], 1, m["tail"])
        return tetra.tetra_gemv(m["codes"], m["row_scales"], s["table"], m["x"], m["y"], m["N"], m["K"])
    if kind == "list":
        tetra.tetra_gemv_list(s["problems"], s["table"])
        return [it["y"] for it in s["items"]]
    if kind == "layer":
        for step in s["steps"]:
            tetra.tetra_gemv_list(step, s["table"])
        return [it["y"] for it in s["items"]]
    if kind == "pass":
        tetra.tetra_gemv_grouped_run(s["ws"], s["table"])
        return s["y"]
    if kind == "batched":
        m = s["m"]
        return tetra.tetra_gemv_batched(m["codes"], m["row_scales"], s["table"], m["x"], m["y"], m["N"], m["K"], s["batch"],
                                        m["tail"], s["ws"])
    if kind == "q4":
        return tetra.tetra_q4_gemv(s["packed"], s["x"], s["y"], s["N"], s["K"], s["G"], s["batch"])
    if kind == "q4list":
        tetra.tetra_q4_list_run(s["ws"], 128)
        return s["y"]
    if kind == "q4rows":
        return tetra.tetra_q4_rows(s["packed"], s["ids"], s["out"], s["N"], s["K"], 64)
    if kind == "encode":
        return tetra.tetra_encode_blocks(s["w"], s["table"], s["sigma"])
    out = []
    for n, B, codes in s["tetra"]:
        out.append(tetra.tetra_decode_packed(tetra.tetra_pack_codes(codes, s["table"], n, B), s["table"], n, B))
    for n, k, source, ids in s["q4"]:
        packed = tetra.tetra_q4_pack(*source, n, k, 128)
        rows = torch.empty((64, k), dtype=torch.float16, device=DEVICE)
        out.append(tetra.tetra_q4_rows(packed, ids, rows, n, k, 128))
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _gemv_bytes(N, K, rule="tail", batch=1):
    blocks = K // 24 if rule == "tail" else -(-K // 24)
    ntail = K % 24 if rule == "tail" else 0
    return N * (6 * blocks + 2 * ntail + 4) + batch * (2 * K + 4 * N)


def _q4_matrix_bytes(N, K, G):
    return N * (K // 2 + 4 * (K // G))


def work(case):
    kind = case["kind"]
    if kind == "gemv":
        return dict(bytes=_gemv_bytes(case["N"], case["K"], case["rule"]), flops=2 * case["N"] * case["K"])
    if kind == "list":
        rows, K = [int(n) for n in case["rows"].split(",")], case["K"]
        return dict(bytes=sum(_gemv_bytes(n, K) for n in rows) - 2 * K * (len(rows) - 1), flops=2 * K * sum(rows))
    if kind in ("layer", "pass"):
        mats = _layer_shapes(case) * case.get("layers", 1)
        return dict(bytes=sum(_gemv_bytes(n, k) for n, k in mats), flops=sum(2 * n * k for n, k in mats))
    if kind == "batched":
        N, K, V = case["N"], case["K"], case["batch"]
        return dict(bytes=_gemv_bytes(N, K, "tail", V), flops=2 * N * K * V)
    if kind == "q4":
        N, K, V = case["N"], case["K"], case["batch"]
        return dict(bytes=_q4_matrix_bytes(N, K, case["G"]) + V * (2 * K + 4 * N), flops=2 * N * K * V)
    if kind == "q4list":
        mats = _int4_shapes(case) * case["layers"]
        return dict(bytes=sum(_q4_matrix_bytes(n, k, 128) + 2 * k + 4 * n for n, k in mats),
                    flops=sum(2 * n * k for n, k in mats))
    if kind == "q4rows":
        K = case["K"]
        return dict(bytes=case["count"] * (4 + K // 2 + 4 * (K // 64) + 2 * K), flops=2 * case["count"] * K)
    if kind == "encode":
        # every trellis path (4096) of both parities has a best point, a sum of 24 products, to be compared
        return dict(bytes=case["blocks"] * (24 * 4 + 4 + 6 + 4), flops=case["blocks"] * 2 * 4096 * 2 * 24)
    total = 0
    for n, k in _layer_shapes(case)[:2] + _layer_shapes(case)[4:6]:
        total += n * (k // 24) * (6 + 24 + 2)                # words in, coordinates, shell and gain out
    for n, k in _int4_shapes(case):
        total += _q4_matrix_bytes(n, k, 128) + 64 * (4 + 2 * k)
    return dict(bytes=total, flops=0)


def tolerance(case):
    if case["kind"] in ("load", "q4rows"):
        return "exact"                       # integers, and float16 values that are one correctly rounded fma each
    if case["kind"] == "encode":
        # the cosine is a sum of 24 float32 products; two points whose cosines agree to that precision are equally good
        return dict(rel=1e-6, max=1e-5, differ=1e-3)
    return dict(rel=1e-5)                    # float32 sums over up to 17,408 terms, most rows far smaller

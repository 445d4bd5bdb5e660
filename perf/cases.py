"""Performance cases: the work that a user of the additive-codebook library has it do.

Decoding (a decoder block's linear layers at 1..16 tokens, replayed from a CUDA graph as a
serving loop does, and single eager calls), prefill (17 tokens to a full 4096-token prompt), the
dense decode of a layer, the per-prefix distortion and the beam-search code update. Shapes are
those of workloads/ (1024^2, 4096^2, the 8B block, 8192^2 with 2^16-entry books, the 70B
up-projection) or drawn around them; codebooks N(0, 0.02^2), codes uniform, scales U(0.5, 1.5),
activations N(0, 1), as in workloads/.
"""
import math

import torch

import paper_2606_12876_gb300 as aq
from paper_2606_12876_gb300.linear import AQLinear, gemv_group

DT = {"f16": torch.float16, "bf16": torch.bfloat16}
DEV = "cuda"


# ------------------------------------------------------------------ cases

def listed():
    block8b = dict(kind="block", hidden=4096, kv=1024, ffn=14336, M=4, B=8, book="f16", x="bf16")
    return [
        # the smallest call: one token through a small layer, issued eagerly (latency and launches)
        dict(name="linear_1024_b1", kind="linear", out=1024, inp=1024, M=2, m=2, B=8, book="f16",
             x="f16", tokens=1),
        # single-stream decoding of an 8B decoder block at full precision (32 bits per group)
        dict(block8b, name="block_b1_m4", m=4, tokens=1),
        # a small serving batch at the deployment's three-codebook precision
        dict(block8b, name="block_b8_m3", m=3, tokens=8),
        # the largest decode batch
        dict(block8b, name="block_b16_m4", m=4, tokens=16),
        # 4-bit codes (16-entry codebooks, the 4x4-bit format), a few concurrent sequences
        dict(block8b, name="block_4bit_b4", B=4, m=4, tokens=4),
        # 2^16-entry codebooks, single-stream
        dict(name="bigbook_8192_b1", kind="linear", out=8192, inp=8192, M=2, m=2, B=16, book="f16",
             x="f16", tokens=1),
        # a short ragged prompt (or a large decode batch) through a down projection
        dict(name="prefill_100_down", kind="linear", out=4096, inp=14336, M=4, m=3, B=8, book="f16",
             x="bf16", tokens=100),
        # an ordinary prompt through a gate projection
        dict(name="prefill_512_gate", kind="linear", out=14336, inp=4096, M=4, m=4, B=8,
             book="f16", x="bf16", tokens=512),
        # a full 4096-token prompt through the 70B up projection
        dict(name="prefill_4096_70b", kind="linear", out=28672, inp=8192, M=4, m=4, B=8,
             book="bf16", x="bf16", tokens=4096),
        # writing a layer out densely for code that wants plain weights
        dict(name="decode_70b_m3", kind="decode", out=28672, inp=8192, M=4, m=3, B=8, book="bf16"),
        # the distortion of every prefix of an attention projection (the training loss)
        dict(name="wmse_4096", kind="wmse", out=4096, inp=4096, M=4, B=8, book="f16"),
        # the code update of a key projection (beam search of width 8)
        dict(name="beam_1024x4096", kind="beam", out=1024, inp=4096, M=4, B=8, book="f16", beam=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dim(rng, lo, hi):
    # a multiple of 8; half of the time a multiple of 256, as most models have
    v = _log(rng, lo, hi)
    return max(lo, v // 256 * 256) if rng.random() < 0.5 else max(lo, v // 8 * 8)


def draw(rng):
    kind = rng.choice(["linear", "linear", "block", "block", "block", "prefill", "prefill", "prefill",
                       "decode", "wmse", "beam"])
    M = rng.randint(2, 5)
    m = rng.randint(1, M)
    book, x = rng.choice(["f16", "f16", "bf16"]), rng.choice(["f16", "bf16"])
    if kind == "linear":
        B = rng.choice([4, 8, 8, 8, 16])
        if B == 16:
            M, m = 2, min(m, 2)
        hi = 8192
        out, inp = _dim(rng, 256, hi), _dim(rng, 256, hi)
        return dict(kind=kind, out=out + rng.choice([0, 0, 3]), inp=inp, M=M, m=m, B=B, book=book, x=x,
                    tokens=1 if B == 16 else rng.randint(1, 16))
    if kind == "block":
        hidden = _dim(rng, 1024, 4096)
        return dict(kind=kind, hidden=hidden, kv=max(8, hidden // 4 // 8 * 8), ffn=_dim(rng, 2048, 14336),
                    M=min(M, 4), m=min(m, 4), B=rng.choice([8, 8, 8, 4]), book=book, x=x,
                    tokens=rng.choice([1, 1, rng.randint(2, 16), rng.randint(2, 16)]))
    if kind == "prefill":
        tokens = _log(rng, 17, 4096)
        out, inp = _dim(rng, 1024, 14336), _dim(rng, 1024, 8192)
        return dict(kind="linear", out=out, inp=inp, M=min(M, 4), m=min(m, 4), B=8, book=book, x=x, tokens=tokens)
    if kind == "decode":
        return dict(kind=kind, out=_dim(rng, 1024, 16384), inp=_dim(rng, 1024, 8192), M=M, m=m,
                    B=rng.choice([8, 8, 4]), book=book)
    if kind == "wmse":
        return dict(kind=kind, out=_dim(rng, 512, 4096), inp=_dim(rng, 512, 4096), M=min(M, 4), B=8, book=book)
    return dict(kind=kind, out=_dim(rng, 256, 1024), inp=_dim(rng, 512, 2048), M=min(M, 4), B=8, book=book,
                beam=rng.choice([1, 2, 4, 8]))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _layer(g, out, inp, M, B, book):
    books = (torch.randn(M, 1 << B, 8, generator=g, device=DEV) * 0.02).to(DT[book])
    codes = torch.randint(0, 1 << B, (out, inp // 8, M), generator=g, device=DEV, dtype=torch.int32)
    scales = (torch.rand(out, generator=g, device=DEV) + 0.5).to(DT[book])
    return dict(out=out, inp=inp, M=M, B=B, book=book, books=books, codes=codes, scales=scales)


def _block_layers(c):
    h, kv, f = c["hidden"], c["kv"], c["ffn"]
    return [(h, h), (kv, h), (kv, h), (h, h), (f, h), (f, h), (h, f)]   # q k v o gate up down


def _inputs(case, seed):
    """Raw inputs of a case: the same for prepare() and exact()."""
    g = _gen(seed)
    k = case["kind"]
    if k == "block":
        layers = [_layer(g, o, i, case["M"], case["B"], case["book"]) for o, i in _block_layers(case)]
        t, dt = case["tokens"], DT[case["x"]]
        xs = [torch.randn(t, n, generator=g, device=DEV).to(dt)
              for n in (case["hidden"], case["hidden"], case["hidden"], case["ffn"])]
        return dict(layers=layers, xs=xs)    # inputs of q/k/v, o, gate/up, down
    L = _layer(g, case["out"], case["inp"], case["M"], case["B"], case["book"])
    if k == "linear":
        x = torch.randn(case["tokens"], case["inp"], generator=g, device=DEV).to(DT[case["x"]])
        return dict(layers=[L], xs=[x])
    if k == "decode":
        return dict(layers=[L], xs=[])
    # wmse, beam: W near the stored reconstruction (a residual-quantized weight), H = X X^T / n
    W = torch.empty(case["out"], case["inp"], device=DEV)
    for r in range(0, case["out"], 1024):
        W[r:r + 1024] = _dense(L, case["M"], r, r + 1024).float()
    W += 0.01 * torch.randn(W.shape, generator=g, device=DEV)
    X = torch.randn(2 * case["inp"], case["inp"], generator=g, device=DEV)
    H = (X.t() @ X) / X.shape[0]
    return dict(layers=[L], xs=[], W=W.to(DT[case["book"]]), H=H)


def _bits(t):
    return t.contiguous().view(torch.int16).cpu().numpy().view("uint16")


def _linear(L):
    codes = L["codes"].to(torch.uint8).cpu().numpy() if L["B"] <= 8 else \
        L["codes"].to(torch.int16).cpu().numpy().view("uint16")
    return AQLinear(_bits(L["books"]), codes, _bits(L["scales"]), L["book"], L["book"], DEV)


_capture_stream = None


def _captured(call):
    """(graph, outputs) of call(), captured after a warm-up on the program's capture stream."""
    global _capture_stream
    if _capture_stream is None:
        _capture_stream = torch.cuda.Stream()
    s = _capture_stream
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        call()
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        out = call()
    return graph, out


def prepare(case, seed):
    d = _inputs(case, seed)
    k = case["kind"]
    st = dict(kind=k, m=case.get("m"))
    if k == "beam":
        # the codes themselves and a fixed workspace, as a training loop keeps them
        L = d["layers"][0]
        layout = aq.Layout.make(L["out"], L["inp"], L["M"], B=L["B"], book_dtype=L["book"], scale_dtype=L["book"])
        st.update(layout=layout, W=d["W"], H=d["H"], books=L["books"], scales=L["scales"],
                  codes=L["codes"].to(torch.uint8).contiguous(), beam=case["beam"], lam=[1.0] * L["M"],
                  ws=aq.workspace(aq.beam_workspace_bytes(layout)))
        return st
    st["layers"] = lins = [_linear(L) for L in d["layers"]]
    st["xs"] = xs = d["xs"]
    if k == "wmse":
        st.update(W=d["W"], H=d["H"], lam=[1.0 / (i + 1) for i in range(case["M"])])
    if k == "block":
        q, kk, v, o, gate, up, down = lins
        m = case["m"]

        def call():
            a = gemv_group([q, kk, v], xs[0], m)
            b = o(xs[1], m)
            c = gemv_group([gate, up], xs[2], m)
            return [*a, b, *c, down(xs[3], m)]
        st["graph"], st["out"] = _captured(call)
    return st


def run(st):
    k = st["kind"]
    if k == "block":
        st["graph"].replay()
        return st["out"]
    if k == "linear":
        return st["layers"][0](st["xs"][0], st["m"])
    if k == "decode":
        return st["layers"][0].decode(st["m"])
    if k == "wmse":
        return st["layers"][0].wmse(st["W"], st["H"], st["lam"])
    out = torch.empty_like(st["codes"])
    aq.aq_beam_search(st["layout"], st["W"], st["codes"], st["books"], st["scales"], st["H"], aq.AQ_F32,
                      st["lam"], st["beam"], out, st["ws"])
    return out


# ------------------------------------------------------------------ what a pass cannot do without

def _weights_bytes(out, inp, m, B):
    return m * (out * (inp // 8) * B // 8 + (16 << B)) + 2 * out


def work(case):
    k, B = case["kind"], case["B"]
    shapes = _block_layers(case) if k == "block" else [(case["out"], case["inp"])]
    if k in ("block", "linear"):
        t = case["tokens"]
        b = sum(_weights_bytes(o, i, case["m"], B) + 2 * t * o for o, i in shapes)
        ins = [case["hidden"]] * 3 + [case["ffn"]] if k == "block" else [case["inp"]]
        return {"bytes": b + 2 * t * sum(ins), "flops": sum(2 * t * o * i for o, i in shapes)}
    out, inp = shapes[0]
    M = case["M"]
    if k == "decode":
        return {"bytes": _weights_bytes(out, inp, case["m"], B) + 2 * out * inp, "flops": out * inp * case["m"]}
    b = _weights_bytes(out, inp, M, B) + 2 * out * inp + 4 * inp * inp
    if k == "wmse":      # H is symmetric in effect: half of E_k H per prefix
        return {"bytes": b + 8 * (M + 1), "flops": M * out * inp * inp}
    # E_k S for every prefix, then per (row, group) a score of at least eight multiply-adds for
    # every (state, codeword) pair
    cand, states = 0, 1
    for _ in range(M):
        cand += states << B
        states = min(case["beam"], states << B)
    return {"bytes": b + M * out * (inp // 8), "flops": 2 * M * out * inp * inp + out * (inp // 8) * cand * 16}


# ------------------------------------------------------------------ 64-bit values

def _dense(L, m, r0=0, r1=None):
    """W_m of rows r0..r1 in 64 bits: s[o] * sum_{k<m} C_k[b_k[o, g]]."""
    r1 = min(L["out"], r1 if r1 is not None else L["out"])
    acc = torch.zeros(r1 - r0, L["inp"] // 8, 8, dtype=torch.float64, device=DEV)
    for k in range(m):
        acc += L["books"][k].double()[L["codes"][r0:r1, :, k].long()]
    return acc.reshape(r1 - r0, L["inp"]) * L["scales"][r0:r1].double()[:, None]


def _product(L, x, m):
    y = torch.empty(x.shape[0], L["out"], dtype=torch.float64, device=DEV)
    for r in range(0, L["out"], 4096):
        y[:, r:r + 4096] = x.double() @ _dense(L, m, r, r + 4096).t()
    return y


def exact(case, seed):
    k = case["kind"]
    if k == "beam":
        return None          # codes: whole numbers
    d = _inputs(case, seed)
    if k == "block":
        which = [0, 0, 0, 1, 2, 2, 3]
        return [_product(L, d["xs"][i], case["m"]) for L, i in zip(d["layers"], which)]
    L = d["layers"][0]
    if k == "linear":
        return _product(L, d["xs"][0], case["m"])
    if k == "decode":
        w = torch.empty(L["out"], L["inp"], dtype=torch.float64, device=DEV)
        for r in range(0, L["out"], 4096):
            w[r:r + 4096] = _dense(L, case["m"], r, r + 4096)
        return w
    H = d["H"].double()
    H = (H + H.t()) / 2
    vals = []
    for p in range(1, case["M"] + 1):
        E = d["W"].double() - _dense(L, p)
        vals.append(((E @ H) * E).sum() / L["out"])
    vals.append(sum(v / (i + 1) for i, v in enumerate(vals)))
    return torch.stack(vals)

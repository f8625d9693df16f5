"""Timing cases of the attention path: calls of the public entry points on the shapes the library is used on.

A case is one layer's problem - a (frames, height, width) token grid with leading text tokens, heads, head dimension,
block geometry - and the call made on it:

    dense      losa_attn                  every warm-up step before the pattern exists
    construct  losa_attn_mass             the one step that builds the pattern (with the rows' log-sum-exp)
    mass       losa_block_mass            the pattern built beside another attention (calibration, analysis)
    select     losa_select / _topk        the pattern itself, from masses in hand; optionally its recall
    sparse     losa_sparse_attn           every later step, on the frozen pattern
    batched    losa_sparse_attn_batched   several small layers or requests in one launch
    chain      mass -> select -> sparse   all three on a layer where launches count

Inputs follow inputs.py's recipe (unit noise plus a shared position component), drawn on the GPU.  The frozen pattern
that `sparse` and `batched` are given is that of a step before: it comes from plain torch on the unperturbed tensors
(masses of a sample of each query block's rows, then the shortest prefix that reaches tau), so that it does not depend
on the code that is timed.
"""
import functools
import math

import torch

import paper_2608_12032_b200 as losa
from paper_2608_12032_b200 import binding, inputs

TAU = 0.99
SAMPLED_ROWS = 32  # rows of a query block whose masses the frozen pattern is built from
MAX_FLOP = 100e12  # dense-equivalent cost of a drawn case; the largest listed one has 173e12


def _case(name, op, grid, n_text, B, H, D, R, C, **more):
    case = {"name": name, "op": op, "t": grid[0], "h": grid[1], "w": grid[2], "n_text": n_text, "B": B, "H": H, "D": D,
            "R": R, "C": C, "layout": "bhnd", "out": "bf16", "layers": 1, "rule": "tau", "recall": False}
    case.update(more)
    return case


def listed():
    small, wan, cog, hunyuan = (8, 16, 16), (21, 30, 52), (13, 30, 45), (33, 45, 80)
    return [
        # the smallest layer, all three calls in a row: launches and host time
        _case("chain_tiny", "chain", (4, 8, 8), 0, 1, 2, 64, 64, 64),
        # a reuse step of a small layer (2048 tokens): a few work items for 148 SMs
        _case("sparse_small", "sparse", small, 0, 1, 4, 64, 64, 64),
        # eight such layers or requests whose inputs are at hand, in one launch
        _case("batched_small_x8", "batched", small, 0, 1, 4, 64, 64, 64, layers=8),
        # a warm-up step of an image-sized layer: both guidance branches, token-major tensors as a projection leaves
        # them, a ragged token count, fp32 output
        _case("dense_ragged_cfg", "dense", (3, 37, 43), 77, 2, 8, 128, 128, 64, layout="bnhd", out="f32"),
        # the paper's three models: CogVideoX-shaped (head dimension 64, 64-row blocks, text tokens first) ...
        _case("dense_cogvideox", "dense", cog, 226, 1, 48, 64, 64, 64),
        _case("sparse_cogvideox", "sparse", cog, 226, 1, 48, 64, 64, 64),
        # ... Wan2.1-shaped, the layer the speedups are quoted on: the construction step and the reuse step
        _case("construct_wan", "construct", wan, 0, 1, 12, 128, 128, 128),
        _case("sparse_wan", "sparse", wan, 0, 1, 12, 128, 128, 128),
        # the same layer with the paper's own block geometry, 128 query rows by 32 keys
        _case("mass_wan_r128c32", "mass", wan, 0, 1, 12, 128, 128, 32),
        _case("sparse_wan_r128c32", "sparse", wan, 0, 1, 12, 128, 128, 32),
        # HunyuanVideo-shaped, the largest: selection over the paper's 32-key blocks, and the reuse step
        _case("select_hunyuan_r128c32", "select", hunyuan, 0, 1, 24, 128, 128, 32),
        _case("sparse_hunyuan", "sparse", hunyuan, 0, 1, 24, 128, 128, 128),
    ]


def draw(rng):
    while True:
        op = rng.choice(["dense", "construct", "mass", "select", "sparse", "sparse", "batched", "chain"])
        D = rng.choice([64, 128])
        R, C = rng.choice([(64, 64), (128, 128), (128, 64), (128, 32)])
        N = math.exp(rng.uniform(math.log(250), math.log(120000)))
        t = rng.randint(1, max(1, min(33, int(N / 64))))
        w = max(4, round(math.sqrt(N / t) * rng.uniform(0.8, 1.25)))
        h = max(4, round(N / (t * w)))
        n_text = rng.choice([0, rng.randint(1, 300)])
        B, H = rng.choice([1, 1, 2]), rng.choice([1, 2, 3, 4, 8, 12, 24, 48])
        layers = rng.randint(2, 8) if op == "batched" else 1
        n = n_text + t * h * w
        tokens = layers * B * H * n
        if 4.0 * tokens * n * D > MAX_FLOP or n > 120000:
            continue
        if tokens * -(-n // C) // R > 1 << 27 or tokens * D > 1 << 29:  # masses of 512 MiB, tensors of 1 GiB
            continue
        if op in ("batched", "chain") and n > 9000:  # small problems: what these two are for
            continue
        case = _case("", op, (t, h, w), n_text, B, H, D, R, C, layout=rng.choice(["bhnd", "bnhd"]),
                     out=rng.choice(["bf16", "bf16", "f32"]), layers=layers, rule=rng.choice(["tau", "tau", "topk"]),
                     recall=op == "select" and rng.random() < 0.5)
        del case["name"]
        return case


def _workload(case):
    return inputs.Workload("case", case["B"], case["H"], case["D"], (case["t"], case["h"], case["w"]), case["n_text"],
                           case["R"], case["C"])


@functools.lru_cache(maxsize=4)
def _position(D, t, h, w, n_text):
    wl = inputs.Workload("case", 1, 1, D, (t, h, w), n_text, 128, 128)
    return inputs.position_component(wl).cuda() * wl.pe_scale


def _qkv(case, seed, layer=0):
    """The layer's q, k of the construction step and q, k, v of the step that is run (bf16, in the case's layout)."""
    B, H, D = case["B"], case["H"], case["D"]
    pe = _position(D, case["t"], case["h"], case["w"], case["n_text"])
    g = torch.Generator("cuda").manual_seed(seed * 64 + layer)
    later = case["op"] in ("sparse", "batched")  # these run at a later step than the one that built the pattern

    def tensor(position):
        x = torch.randn((B, H, pe.shape[0], D), generator=g, device="cuda")
        if position:
            x += pe
        y = x + 0.05 * x.square().mean().sqrt() * torch.randn(x.shape, generator=g, device="cuda") if later else x
        first, now = x.bfloat16(), y.bfloat16()
        if case["layout"] == "bnhd":
            now = now.transpose(1, 2).contiguous().transpose(1, 2)
        return first, now

    (q0, q), (k0, k), (_, v) = tensor(True), tensor(True), tensor(False)
    return q0, k0, q, k, v


def _sampled_mass(case, q, k):
    """[B, H, nQb, nKb] fp32 block masses over a sample of each query block's rows; rows sum to 1."""
    B, H, N, D = q.shape
    R, C = case["R"], case["C"]
    nQb, nKb = -(-N // R), -(-N // C)
    at = torch.arange(nQb, device="cuda")[:, None] * R + torch.arange(SAMPLED_ROWS, device="cuda") * (R // SAMPLED_ROWS)
    at = at.clamp_(max=N - 1)
    mass = torch.empty((B, H, nQb, nKb), device="cuda")
    step = max(1, (1 << 28) // (SAMPLED_ROWS * N))
    for b in range(B):
        for h in range(H):
            for i in range(0, nQb, step):
                rows = at[i:i + step]
                p = torch.softmax((q[b, h, rows.reshape(-1)] @ k[b, h].T).float() / math.sqrt(D), dim=-1)
                p = torch.nn.functional.pad(p.view(*rows.shape, N).mean(1), (0, nKb * C - N))
                mass[b, h, i:i + step] = p.view(-1, nKb, C).sum(-1)
    return mass


def _kept(mass, tau=TAU):
    """Boolean [B, H, nQb, nKb]: the shortest prefix of the sorted masses that reaches tau."""
    value, order = torch.sort(mass, dim=-1, descending=True, stable=True)
    value = value.double()
    keep = torch.cumsum(value, -1) - value < tau
    return torch.zeros_like(keep).scatter_(-1, order, keep)


def _csr(keep):
    rows = keep.reshape(-1, keep.shape[-1])
    offsets = torch.zeros(rows.shape[0] + 1, dtype=torch.int32, device="cuda")
    offsets[1:] = torch.cumsum(rows.sum(1), 0)
    return offsets, rows.nonzero()[:, 1].int()


def _pattern(case, q0, k0):
    return _csr(_kept(_sampled_mass(case, q0, k0)))


def _workspace(op, q, case):
    need = losa.losa_workspace_bytes(op, losa.make_problem(q, case["R"], case["C"]))
    return torch.empty(max(need, 1), dtype=torch.uint8, device="cuda")


def _topk(nKb):
    return max(1, (2 * nKb) // 3)  # about the share of blocks that tau keeps


def prepare(case, seed):
    op, R, C = case["op"], case["R"], case["C"]
    dtype = torch.bfloat16 if case["out"] == "bf16" else torch.float32
    q0, k0, q, k, v = _qkv(case, seed)
    B, H, N, _ = q.shape
    nQb, nKb = -(-N // R), -(-N // C)
    rows = B * H * nQb
    s = {"op": op, "R": R, "C": C, "q": q, "k": k, "v": v, "rule": case["rule"], "topk": _topk(nKb), "recall": case["recall"]}
    if op in ("dense", "construct", "sparse", "chain"):
        s["o"] = torch.empty_strided(q.shape, q.stride(), dtype=dtype, device="cuda")
    if op in ("construct", "mass", "chain"):
        s["mass"] = torch.empty((B, H, nQb, nKb), dtype=torch.float32, device="cuda")
    if op in ("select", "chain"):
        room = rows * (s["topk"] if case["rule"] == "topk" else nKb)
        s["csr"] = (torch.zeros(rows + 1, dtype=torch.int32, device="cuda"), torch.zeros(room, dtype=torch.int32, device="cuda"))
        s["ws_select"] = _workspace(binding.LOSA_OP_SELECT, q, case)
    if op == "dense":
        s["ws"] = _workspace(binding.LOSA_OP_ATTN, q, case)
    elif op == "construct":
        s["ws"] = _workspace(binding.LOSA_OP_ATTN_MASS, q, case)
    elif op == "select":
        s["mass"] = _sampled_mass(case, q0, k0)
        s["q"] = s["k"] = s["v"] = None
    elif op == "sparse":
        s["ws"] = _workspace(binding.LOSA_OP_SPARSE_ATTN, q, case)
        s["pattern"] = _pattern(case, q0, k0)
    elif op == "batched":
        s["layers"], s["outs"] = [], []
        for i in range(case["layers"]):
            q0, k0, q, k, v = _qkv(case, seed, i)
            s["layers"].append((q, k, v, *_pattern(case, q0, k0)))
            s["outs"].append(torch.empty_strided(q.shape, q.stride(), dtype=dtype, device="cuda"))
        need = binding.losa_workspace_bytes_batched(binding.LOSA_OP_SPARSE_ATTN, losa.make_problem(q, R, C), case["layers"])
        s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    if op in ("mass", "chain"):
        s["ws_mass"] = _workspace(binding.LOSA_OP_BLOCK_MASS, q, case)
    if op == "chain":
        s["ws"] = _workspace(binding.LOSA_OP_SPARSE_ATTN, q, case)
    return s


def _select(s, mass):
    if s["rule"] == "topk":
        return losa.losa_select_topk(mass, s["topk"], ws=s["ws_select"])
    return losa.losa_select(mass, TAU, ws=s["ws_select"], out=s["csr"])


def run(s):
    op, R, C = s["op"], s["R"], s["C"]
    if op == "dense":
        return losa.losa_attn(s["q"], s["k"], s["v"], R, C, out_dtype=s["o"].dtype, out=s["o"], ws=s["ws"])
    if op == "construct":
        return losa.losa_attn_mass(s["q"], s["k"], s["v"], R, C, return_lse=True, out=s["o"], mass=s["mass"], ws=s["ws"])
    if op == "mass":
        return losa.losa_block_mass(s["q"], s["k"], R, C, ws=s["ws_mass"], mass=s["mass"])
    if op == "select":
        csr = _select(s, s["mass"])
        return csr + losa.losa_row_recall(s["mass"], *csr) if s["recall"] else csr
    if op == "sparse":
        return losa.losa_sparse_attn(s["q"], s["k"], s["v"], *s["pattern"], R, C, out=s["o"], ws=s["ws"])
    if op == "batched":
        return losa.losa_sparse_attn_batched(s["layers"], R, C, outs=s["outs"], ws=s["ws"])
    mass = losa.losa_block_mass(s["q"], s["k"], R, C, ws=s["ws_mass"], mass=s["mass"])
    csr = _select(s, mass)
    return mass, losa.losa_sparse_attn(s["q"], s["k"], s["v"], *csr, R, C, out=s["o"], ws=s["ws"])


@functools.lru_cache(maxsize=64)
def _pairs(items):
    """(query, key) token pairs the frozen pattern keeps and its list entries: of one seed, they hardly change with it."""
    case = dict(items)
    q0, k0, *_ = _qkv(case, 1)
    keep = _kept(_sampled_mass(case, q0, k0))
    return float((_tokens(q0.shape[2], case["R"])[:, None] * _tokens(q0.shape[2], case["C"]) * keep).sum()), int(keep.sum())


def _tokens(N, block):
    size = torch.full((-(-N // block),), float(block), device="cuda", dtype=torch.float64)
    size[-1] = N - (len(size) - 1) * block
    return size


def work(case):
    wl = _workload(case)
    B, H, N, D, op, L = wl.B, wl.H, wl.N, wl.D, case["op"], case["layers"]
    tensor, o = B * H * N * D * 2, B * H * N * D * (2 if case["out"] == "bf16" else 4)
    mass, square = 4 * wl.rows * wl.nKb, float(B * H) * N * N
    key = tuple(sorted({**case, "name": "", "op": "sparse"}.items()))
    if op == "dense":
        return {"bytes": 3 * tensor + o, "flops": 4 * D * square}
    if op == "construct":
        return {"bytes": 3 * tensor + o + mass + 4 * B * H * N, "flops": 4 * D * square}
    if op == "mass":
        return {"bytes": 2 * tensor + mass, "flops": 2 * D * square}
    pairs, nnz = _pairs(key)
    if case["rule"] == "topk" and op in ("select", "chain"):
        nnz = wl.rows * _topk(wl.nKb)
        pairs = square * _topk(wl.nKb) / wl.nKb
    csr = 4 * (nnz + wl.rows + 1)
    if op == "select":
        return {"bytes": mass + csr + (16 * wl.rows if case["recall"] else 0), "flops": wl.rows * wl.nKb}
    if op == "chain":
        return {"bytes": 3 * tensor + o + mass + csr, "flops": 2 * D * square + 4 * D * pairs}
    return {"bytes": L * (3 * tensor + o + csr), "flops": L * 4 * D * pairs}


def tolerance(case):
    if case["op"] == "select":
        return {"rel": 1e-12} if case["recall"] else "exact"
    if case["op"] == "mass":
        return {"rel": 5e-6}
    return {"rel": 1e-2, "max": 0.5}


def _attention64(q, k, v, R, C, keep=None, want_mass=False):
    """(o, mass, lse) of softmax attention in fp64, over the kept blocks only where `keep` [B, H, nQb, nKb] is given."""
    B, H, N, D = q.shape
    nQb, nKb = -(-N // R), -(-N // C)
    o = torch.empty((B, H, N, D), device="cuda", dtype=torch.float64)
    mass = torch.empty((B, H, nQb, nKb), device="cuda", dtype=torch.float64)
    lse = torch.empty((B, H, N), device="cuda", dtype=torch.float64)
    step = max(1, (1 << 28) // (N * R))
    for b in range(B):
        for h in range(H):
            kk = k[b, h].double().T.contiguous()
            vv = v[b, h].double() if v is not None else None
            for i in range(0, nQb, step):
                rows = slice(i * R, min(N, (i + step) * R))
                x = q[b, h, rows].double() @ kk
                x /= math.sqrt(D)
                if keep is not None:
                    gone = ~keep[b, h, i:i + step].repeat_interleave(C, 1)[:, :N]
                    x.masked_fill_(gone.repeat_interleave(R, 0)[:x.shape[0]], -math.inf)
                top = x.amax(1, keepdim=True)
                x.sub_(top).exp_()
                total = x.sum(1, keepdim=True)
                lse[b, h, rows] = (top + total.log())[:, 0]
                if vv is not None:
                    o[b, h, rows] = (x @ vv).div_(total)
                if want_mass:
                    x.div_(total)
                    for n, at in enumerate(range(0, x.shape[0], R)):
                        part = torch.nn.functional.pad(x[at:at + R].mean(0), (0, nKb * C - N))
                        mass[b, h, i + n] = part.view(nKb, C).sum(1)
    return o, mass, lse


def _kept_topk(mass, k):
    order = torch.sort(mass, dim=-1, descending=True, stable=True)[1]
    return torch.zeros(mass.shape, dtype=torch.bool, device="cuda").scatter_(-1, order[..., :k], True)


def exact(case, seed):
    op, R, C = case["op"], case["R"], case["C"]
    q0, k0, q, k, v = _qkv(case, seed)
    if op == "dense":
        return _attention64(q, k, v, R, C)[0]
    if op == "construct":
        return _attention64(q, k, v, R, C, want_mass=True)
    if op == "mass":
        return _attention64(q, k, None, R, C, want_mass=True)[1]
    if op == "select":
        if not case["recall"]:
            return None
        mass = _sampled_mass(case, q0, k0)
        keep = _kept_topk(mass, _topk(mass.shape[-1])) if case["rule"] == "topk" else _kept(mass)
        mass = mass.double()
        return None, None, (mass * keep).sum(-1).reshape(-1), mass.sum(-1).reshape(-1)
    if op == "sparse":
        return _attention64(q, k, v, R, C, keep=_kept(_sampled_mass(case, q0, k0)))[0]
    if op == "batched":
        outs = []
        for i in range(case["layers"]):
            q0, k0, q, k, v = _qkv(case, seed, i)
            outs.append(_attention64(q, k, v, R, C, keep=_kept(_sampled_mass(case, q0, k0)))[0])
        return outs
    mass = _attention64(q, k, None, R, C, want_mass=True)[1]
    keep = _kept_topk(mass, _topk(mass.shape[-1])) if case["rule"] == "topk" else _kept(mass)
    return mass, _attention64(q, k, v, R, C, keep=keep)[0]

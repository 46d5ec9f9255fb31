"""The work a user of this library has it do, as measurable cases.

One case is one call (or one drafting round) through the public entry points of
`paper_2609_37029_gb300.lsp`:

  round     lsp_view_update + lsp_draft, captured once as a CUDA graph and
            replayed, which is how a serving loop and bench.py run it
  fold      lsp_view_update of a chunk of prefix rows (chunked prefill: the only
            way to build the summary of an fp32 state, or of rows that arrive in
            pieces), the interface then exported to host memory
  prefill   lsp_prefill of one request's whole prefix, the interface exported to
            host memory (the target side hands it to the drafting side)
  sample    lsp_sample (state workspace) or lsp_sample_noalloc (`noalloc`)
  verify    lsp_verify: acceptance of the drafted blocks
  linear    lsp_linear: one projection

Shapes come from the five workloads of `synth.py`, from the tests and from
bench.py (the paper's B = 7, its ablation variants).
"""
from __future__ import annotations

import math
import weakref

import torch

from paper_2609_37029_gb300 import lsp, synth

DEV = "cuda"
SEED = 7            # key of the sampler's random stream
EPS, THETA = 1.0e-6, 1.0e6


def listed():
    q8b = dict(L=5, H=4096, nq=32, nkv=8, d=128, F=12288, V=151936, W=256, R=16, rc=64, dtype="bf16")
    return [
        # the smallest configuration end to end: one request, one fp32 layer, greedy; launches and latency
        dict(name="round-tiny", kind="round", C=1, B=8, L=3, D=1, H=256, nq=4, nkv=2, d=64, F=1024, V=1024,
             W=256, R=16, rc=64, dtype="f32", t=2048, rows=8, temperature=0.0),
        # the headline: a serving batch of 16 requests, sampled, behind a 32K prefix
        dict(name="round-qwen3-8b", kind="round", C=16, B=16, D=5, t=32768, rows=16, temperature=1.0, **q8b),
        # chunked prefill: two requests' next 2048-row chunk, one of them ragged
        dict(name="fold-chunk", kind="fold", C=2, t=8192, rows=2048, **q8b),
        # the longest prefix of the paper's sweep, built in one call
        dict(name="prefill-128k", kind="prefill", t=131072, **q8b),
        # a short prompt with an odd row count on the large shape's heads (five query heads a KV head)
        dict(name="prefill-1999", kind="prefill", t=1999, **{**q8b, "H": 5120, "nq": 40, "F": 17408}),
        # proposal sampling on its own for a full batch, with the verification logits
        dict(name="sample-c16", kind="sample", noalloc=False, C=16, B=16, V=151936, rc=64, dtype="bf16", temperature=1.0),
        # the paper's block of 7 for a few requests under another framework's allocator, cooler sampling
        dict(name="sample-noalloc-b7", kind="sample", noalloc=True, C=5, B=7, V=151936, rc=64, dtype="bf16", temperature=0.7),
        # acceptance of a full batch's blocks, sampled
        dict(name="verify-c16", kind="verify", C=16, B=16, V=151936, temperature=1.0),
        # greedy acceptance for a few requests with a small vocabulary
        dict(name="verify-greedy-c4", kind="verify", C=4, B=16, V=32000, temperature=0.0),
        # the vocabulary head of a full batch: the largest projection
        dict(name="linear-head-m256", kind="linear", M=256, N=151936, K=4096, splits=1, dtype="bf16"),
        # the MLP down projection for one request's block of 7
        dict(name="linear-down-m7", kind="linear", M=7, N=4096, K=12288, splits=9, dtype="bf16"),
        # the gate projection of the large shape's 32 x 16 tokens
        dict(name="linear-gate-m512", kind="linear", M=512, N=17408, K=5120, splits=1, dtype="bf16"),
    ]


# ------------------------------------------------------------------ more cases of the same ranges
def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _log_mult(rng, lo, hi, step):
    return max(lo, _log(rng, lo, hi) // step * step)


# (H, nq, nkv, F, V) of the bf16 workloads, head dim 128
_WIDTHS = [(1024, 8, 2, 4096, 32000), (4096, 32, 8, 12288, 151936), (5120, 40, 8, 17408, 151936)]


def draw(rng):
    kind = rng.choice(["round", "fold", "prefill", "sample", "verify", "linear", "linear"])
    H, nq, nkv, F, V = rng.choice(_WIDTHS)
    heads = dict(L=rng.randint(2, 5), H=H, nq=nq, nkv=nkv, d=128, F=F, V=V, W=rng.choice([64, 128, 256]),
                 R=rng.choice([8, 16]), rc=64, dtype="bf16")
    temperature = rng.choice([0.0, 0.7, 1.0])
    if kind == "round":
        case = dict(kind=kind, C=rng.randint(1, 16), B=rng.randint(4, 16), t=_log(rng, 1, 131072),
                    rows=rng.randint(1, 17), temperature=temperature, **heads)
        if H != 5120 and rng.random() < 0.3:      # the fp32 reference path: small widths only
            case.update(dtype="f32", d=64, H=256, nq=4, nkv=2, F=1024, V=1024, C=rng.randint(1, 8))
        case["D"] = min(case["L"], rng.randint(1, 3))
        return case
    if kind == "fold":
        return dict(kind=kind, C=rng.randint(1, 4), t=_log(rng, 1, 131072), rows=_log(rng, 1, 4096), **heads)
    if kind == "prefill":
        return dict(kind=kind, t=_log(rng, 1, 131072), **heads)
    if kind == "sample":
        return dict(kind=kind, noalloc=rng.random() < 0.5, C=_log(rng, 1, 32), B=rng.randint(4, 16),
                    V=_log_mult(rng, 1024, 151936, 16), rc=rng.choice([32, 64]), dtype="bf16", temperature=temperature)
    if kind == "verify":
        return dict(kind=kind, C=_log(rng, 1, 32), B=rng.randint(4, 16), V=_log_mult(rng, 1024, 151936, 16),
                    temperature=temperature)
    case = dict(kind=kind, M=_log(rng, 1, 512), N=_log(rng, 500, 40000), K=_log_mult(rng, 256, 20480, 8),
                dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]))
    case["splits"] = rng.randint(1, max(1, min(9, case["K"] // 512)))
    return case


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _randn(g, *shape, std=1.0, dtype=torch.float32):
    x = torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)
    return (x.mul_(std) if std != 1.0 else x).to(dtype)


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _shape(case):
    """The configuration a case runs under; sizes it does not touch are the smallest allowed."""
    get = case.get
    return synth.LspShape("case", C=get("C", 1), B=get("B", 16), L=get("L", 1), D=get("D", 1), H=get("H", 128),
                          nq=get("nq", 1), nkv=get("nkv", 1), d=get("d", 128), F=get("F", 64), V=get("V", 1024),
                          W=get("W", 16), R=get("R", 16), rc=get("rc", 64), dtype=get("dtype", "bf16"),
                          rope_theta=THETA, rms_eps=EPS)


def _parts(s):
    """The exported interface's tensors in order: (name, shape, dtype)."""
    dt = s.torch_dtype
    return [("win_k", (s.C, s.L, s.nkv, s.W, s.d), dt), ("win_v", (s.C, s.L, s.nkv, s.W, s.d), dt),
            ("m", (s.C, s.L, s.nq, s.R, s.d), torch.float32), ("eta", (s.C, s.L, s.nq, s.R), torch.float32),
            ("h", (s.C, s.L, s.H), dt), ("t", (s.C,), torch.int64)]


def _interface_buffer(s):
    """A pinned host buffer for lsp_state_export / import and its tensors by name."""
    buf = torch.empty(lsp.lsp_state_bytes(lsp.make_config(s)), dtype=torch.uint8, pin_memory=True)
    views, off = {}, 0
    for name, shape, dt in _parts(s):
        n = math.prod(shape) * torch.empty((), dtype=dt).element_size()
        views[name] = buf[off:off + n].view(dt).view(shape)
        off += n
    return buf, views


def _interface(g, s, t):
    """The interface a prefix of t rows leaves behind: a full ring of the last rows (zeros where
    t < W), summary values that are averages over many rows, the log-normaliser of t rows."""
    dt = s.torch_dtype
    st = {"win_k": _randn(g, s.C, s.L, s.nkv, s.W, s.d, dtype=dt), "win_v": _randn(g, s.C, s.L, s.nkv, s.W, s.d, dtype=dt),
          "m": _randn(g, s.C, s.L, s.nq, s.R, s.d, std=1.6 / math.sqrt(t + 1.0)),
          "eta": _randn(g, s.C, s.L, s.nq, s.R, std=0.1) + (math.log(t) + 0.5),
          "h": _randn(g, s.C, s.L, s.H, dtype=dt), "t": torch.full((s.C,), t, dtype=torch.int64, device=DEV)}
    if t < s.W:
        st["win_k"][:, :, :, t:] = 0
        st["win_v"][:, :, :, t:] = 0
    return st


def _target_rows(g, s, rows):
    """(k, v, h) of `rows` new target rows per request, h of the boundary row only."""
    dt = s.torch_dtype
    return (_randn(g, s.C, s.L, rows, s.nkv, s.d, dtype=dt), _randn(g, s.C, s.L, rows, s.nkv, s.d, dtype=dt),
            _randn(g, s.C, s.L, 1, s.H, dtype=dt))


def _accepted(g, s, rows, lo):
    acc = torch.randint(lo, rows + 1, (s.C,), generator=g, device=DEV, dtype=torch.int32)
    acc[0] = rows
    return acc


def _logits(g, case):
    """Target and draft logits of a block and the tokens the drafter drew from its own."""
    C, B, V, T = case["C"], case["B"], case["V"], case["temperature"]
    zt = _randn(g, C, B + 1, V, std=2.0)
    a = 0.9 + 0.099 * torch.rand(C, 1, 1, generator=g, device=DEV)
    zq = a * zt[:, :B] + torch.sqrt(1 - a * a) * _randn(g, C, B, V, std=2.0)
    score = zq if T == 0 else zq / T - torch.log(-torch.log(torch.rand(C, B, V, generator=g, device=DEV).clamp_(1e-9, 1 - 1e-7)))
    return zt, zq.contiguous(), score.argmax(-1).to(torch.int32).contiguous()


def _inputs(case, seed):
    """Every tensor of a case, from the seed alone."""
    g, s, kind = _gen(seed), _shape(case), case["kind"]
    x = {}
    if kind == "round":
        x["w"] = synth.make_weights(s, seed=seed, device=DEV)
        x["state"] = _interface(g, s, case["t"])
        x["k"], x["v"], x["h"] = _target_rows(g, s, case["rows"])
        x["acc"] = _accepted(g, s, case["rows"], 1)
        x["block"] = torch.full((s.C, s.B), -1, dtype=torch.int32, device=DEV)
        x["block"][:, 0] = torch.randint(0, s.V, (s.C,), generator=g, device=DEV, dtype=torch.int32)
    elif kind == "fold":
        x["G"] = _randn(g, s.L, s.nq, s.R, s.d, std=s.d ** -0.5, dtype=s.torch_dtype)
        x["state"] = _interface(g, s, case["t"])
        x["k"], x["v"], x["h"] = _target_rows(g, s, case["rows"])
        x["acc"] = _accepted(g, s, case["rows"], (case["rows"] + 1) // 2)
    elif kind == "prefill":
        x["G"] = _randn(g, s.L, s.nq, s.R, s.d, std=s.d ** -0.5, dtype=s.torch_dtype)
        for n in ("k", "v"):
            x[n] = torch.stack([_randn(g, case["t"], s.nkv, s.d, dtype=s.torch_dtype) for _ in range(s.L)])
        x["h"] = _randn(g, s.L, 1, s.H, dtype=s.torch_dtype)
    elif kind == "sample":
        x["z"] = _randn(g, s.C, s.B, s.V, std=1.5)
        x["prev"] = torch.randint(0, s.V, (s.C,), generator=g, device=DEV, dtype=torch.int32)
        x["Ec"], x["Wc"] = (_randn(g, s.V, s.rc, std=0.1, dtype=s.torch_dtype) for _ in range(2))
    elif kind == "verify":
        x["zt"], x["zq"], x["y"] = _logits(g, case)
    else:
        x["x"] = _randn(g, case["M"], case["K"], dtype=_dtype(case))
        x["w"] = _randn(g, case["N"], case["K"], std=0.02, dtype=_dtype(case))
    return x


# ------------------------------------------------------------------ what a program keeps, and one pass
class Session:
    """A library state with the buffers of one case; freed with the object."""

    def __init__(self, case, x):
        self.case, self.x, self.shape, self.graph = case, x, _shape(case), None
        self.st = None
        s, kind = self.shape, case["kind"]
        if kind in ("round", "fold", "prefill", "verify") or (kind == "sample" and not case["noalloc"]):
            self.st = lsp.lsp_state_create(lsp.make_config(s))
            weakref.finalize(self, lsp.lsp_state_destroy, self.st)
        if kind in ("round", "fold", "prefill"):
            G = x["w"]["G"] if kind == "round" else x["G"]
            lsp.lsp_state_init(self.st, G)
            self.buf, self.views = _interface_buffer(s)
        if kind == "fold":
            self.restore()
        if kind in ("round", "sample"):
            self.sp = lsp.make_sample_params(case["temperature"], SEED, 3)
            self.tokens = torch.empty(s.C, s.B, dtype=torch.int32, device=DEV)
            self.logits = torch.empty(s.C, s.B, s.V, device=DEV)
        if kind == "round":
            self.weights = lsp.make_weights(x["w"])
            self.round()                            # plans are laid out once, before the capture
            self.restore()
            torch.cuda.synchronize()
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph):
                self.round()
        if kind == "verify":
            self.sp = lsp.make_sample_params(case["temperature"], SEED, 3)
            self.accepted = torch.empty(s.C, dtype=torch.int32, device=DEV)
            self.next = torch.empty(s.C, dtype=torch.int32, device=DEV)
        if kind == "linear":
            self.y = torch.empty(case["M"], case["N"], device=DEV)
            self.ws_bytes = lsp.lsp_linear_workspace_bytes(case["M"], case["N"], case["splits"])
            self.ws = torch.empty(max(16, self.ws_bytes), dtype=torch.uint8, device=DEV)

    def restore(self):
        """The prefix's interface into the state."""
        for n, v in self.x["state"].items():
            self.views[n].copy_(v)
        torch.cuda.synchronize()
        lsp.lsp_state_import(self.st, self.buf)

    def round(self):
        x = self.x
        lsp.lsp_view_update(self.st, x["k"], x["v"], x["h"], x["acc"], h_rows=1)
        lsp.lsp_draft(self.st, x["block"], self.weights, self.sp, self.tokens, self.logits)


def prepare(case, seed):
    return Session(case, _inputs(case, seed))


def run(state):
    x, case, kind, s = state.x, state.case, state.case["kind"], state.shape
    if kind == "round":
        state.graph.replay()
        return {"tokens": state.tokens, "logits": state.logits}
    if kind in ("fold", "prefill"):
        if kind == "fold":
            lsp.lsp_view_update(state.st, x["k"], x["v"], x["h"], x["acc"], h_rows=1)
        else:
            lsp.lsp_prefill(state.st, 0, x["k"], x["v"], x["h"], h_rows=1)
        lsp.lsp_state_export(state.st, state.buf)
        return state.views
    if kind == "sample":
        if case["noalloc"]:
            lsp.lsp_sample_noalloc(x["z"], x["prev"], x["Ec"], x["Wc"], lsp.LSP_DTYPE_BF16, s.C, s.B, s.V, s.rc, state.sp,
                                   state.tokens, state.logits)
        else:
            lsp.lsp_sample(state.st, x["z"], x["prev"], x["Ec"], x["Wc"], state.sp, state.tokens, state.logits)
        return {"tokens": state.tokens, "logits": state.logits}
    if kind == "verify":
        lsp.lsp_verify(state.st, x["zt"], x["zq"], x["y"], state.sp, state.accepted, state.next)
        return {"accepted": state.accepted, "next": state.next}
    dt = lsp.LSP_DTYPE_BF16 if case["dtype"] == "bf16" else lsp.LSP_DTYPE_F32
    lsp.lsp_linear(x["x"], x["w"], state.y, case["M"], case["N"], case["K"], dt, case["splits"], state.ws, state.ws_bytes)
    return state.y


# ------------------------------------------------------------------ the least a pass has to do
def work(case):
    kind, s = case["kind"], _shape(case)
    es = 2 if s.dtype == "bf16" else 4
    iface = lsp.lsp_state_bytes(lsp.make_config(s))
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": (M + N) * K * es + 4 * M * N, "flops": 2 * M * N * K}
    if kind == "verify":
        C, B, V = case["C"], case["B"], case["V"]
        rows = 2 * B + 1 if case["temperature"] > 0 else B + 1       # target rows, and the draft rows when sampling
        return {"bytes": 4 * C * rows * V + 8 * C, "flops": C * rows * V}
    table = s.C * s.B * s.V
    if kind == "sample":
        return {"bytes": 2 * 4 * table + min(s.V, s.C * s.B) * s.rc * es + s.V * s.rc * es, "flops": 2 * table * s.rc}
    row = 2 * s.L * s.nkv * s.d * es                                 # K and V of one prefix row
    if kind == "prefill":
        return {"bytes": case["t"] * row + 2 * iface, "flops": 4 * case["t"] * s.L * s.nq * s.R * s.d}
    if kind == "fold":
        n = 0.75 * s.C * case["rows"]
        return {"bytes": n * row + 3 * iface, "flops": 4 * n * s.L * s.nq * s.R * s.d}
    M, qkv = s.M, (s.nq + 2 * s.nkv) * s.d
    per_layer = s.H * qkv + s.nq * s.d * s.H + 3 * s.F * s.H
    mats = s.D * per_layer + s.V * s.H
    context = s.D * s.C * (s.B + s.W + s.R) * s.nq * s.B * s.d
    bytes_ = (mats + s.L * s.H * s.H + M * s.H + 2 * s.V * s.rc) * es + 4 * table
    bytes_ += 0.5 * s.C * case["rows"] * row + 2 * iface
    return {"bytes": bytes_, "flops": 2 * M * mats + 2 * s.C * s.L * s.H * s.H + 4 * context + 2 * table * s.rc}


# ------------------------------------------------------------------ the same results in 64 bits
def _fold64(s, G, state, k, v, h, acc):
    """The interface after folding acc[b] rows: (win_k, win_v, m, eta, h) in fp64."""
    out = {n: state[n].double().clone() for n in ("win_k", "win_v", "m", "eta", "h")}
    rep = s.nq // s.nkv
    for b in range(s.C):
        n, t = int(acc[b]), int(state["t"][b])
        for l in range(s.L):
            for g in range(s.nkv):
                kg, vg = k[b, l, :n, g].double(), v[b, l, :n, g].double()
                q = G[l, g * rep:(g + 1) * rep].double().reshape(rep * s.R, s.d)
                sc = q @ kg.T / math.sqrt(s.d)
                en = torch.logsumexp(sc, 1)
                mn = torch.exp(sc - en[:, None]) @ vg
                heads = (b, l, slice(g * rep, (g + 1) * rep))
                ea, ma = out["eta"][heads].reshape(-1), out["m"][heads].reshape(rep * s.R, s.d)
                e = torch.logaddexp(ea, en)
                out["m"][heads] = (torch.exp(ea - e)[:, None] * ma + torch.exp(en - e)[:, None] * mn).view(rep, s.R, s.d)
                out["eta"][heads] = e.view(rep, s.R)
            keep = min(n, s.W)
            if keep:
                slots = torch.arange(t + n - keep, t + n, device=DEV) % s.W
                out["win_k"][b, l, :, slots] = k[b, l, n - keep:n].double().transpose(0, 1)
                out["win_v"][b, l, :, slots] = v[b, l, n - keep:n].double().transpose(0, 1)
            out["h"][b, l] = h[b, l, -1].double()
    return out


def _norm64(x, w):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS) * w.double()


def _rope64(x, pos):
    half = x.shape[-1] // 2
    ang = pos.double()[:, None] * THETA ** (-2.0 * torch.arange(half, device=DEV, dtype=torch.float64) / x.shape[-1])
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)


def _base64(s, w, f, t, block):
    """Base logits [C][B][V] of one drafter forward over the interface f, in fp64."""
    rep, C, B = s.nq // s.nkv, s.C, s.B
    emb = torch.where((block >= 0)[..., None], w["embed"][block.clamp(min=0).long()].double(), w["mask_emb"].double())
    x = emb + w["pos"].double() + (f["h"].reshape(C, -1) @ w["fuse"].double().T)[:, None]
    pos = (t[:, None] + torch.arange(B, device=DEV)).reshape(-1)
    for j, lw in enumerate(w["layers"]):
        l = s.layer_map[j]
        xn = _norm64(x, lw["in_norm"]).reshape(C * B, s.H)
        q = _rope64(_norm64((xn @ lw["wq"].double().T).view(-1, s.nq, s.d), lw["q_norm"]), pos).view(C, B, s.nq, s.d)
        k = _rope64(_norm64((xn @ lw["wk"].double().T).view(-1, s.nkv, s.d), lw["k_norm"]), pos).view(C, B, s.nkv, s.d)
        v = (xn @ lw["wv"].double().T).view(C, B, s.nkv, s.d)
        o = torch.empty(C, B, s.nq, s.d, device=DEV, dtype=torch.float64)
        for b in range(C):
            n = min(int(t[b]), s.W)
            for h in range(s.nq):
                g = h // rep
                keys = torch.cat([k[b, :, g], f["win_k"][b, l, g, :n], w["G"][l, h].double()])
                vals = torch.cat([v[b, :, g], f["win_v"][b, l, g, :n], f["m"][b, l, h]])
                o[b, :, h] = torch.softmax(q[b, :, h] @ keys.T / math.sqrt(s.d), -1) @ vals
        x = x + (o.reshape(C * B, -1) @ lw["wo"].double().T).view(C, B, s.H)
        xn = _norm64(x, lw["post_norm"]).reshape(C * B, s.H)
        up = torch.nn.functional.silu(xn @ lw["w_gate"].double().T) * (xn @ lw["w_up"].double().T)
        x = x + (up @ lw["w_down"].double().T).view(C, B, s.H)
    xn = _norm64(x, w["final_norm"]).reshape(C * B, s.H)
    z = torch.empty(C * B, s.V, device=DEV, dtype=torch.float64)
    for v0 in range(0, s.V, 16384):
        z[:, v0:v0 + 16384] = xn @ w["lm_head"][v0:v0 + 16384].double().T
    return z.view(C, B, s.V)


def _gumbel64(C, V, step, rnd):
    """-log(-log u) with u from Philox4x32-10 (Salmon et al., SC'11) at counter (v >> 2, step, b, rnd)."""
    mask = 0xFFFFFFFF
    c = [torch.arange((V + 3) // 4, device=DEV)[None].expand(C, -1), torch.full((C, 1), step, device=DEV),
         torch.arange(C, device=DEV)[:, None], torch.full((C, 1), rnd, device=DEV)]
    k0, k1 = SEED & mask, SEED >> 32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57                  # low 64 bits of the 32 x 32 products
        c = [((b >> 32) & mask) ^ c[1] ^ k0, b & mask, ((a >> 32) & mask) ^ c[3] ^ k1, a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    words = torch.stack([x.expand(C, (V + 3) // 4) for x in c], -1).reshape(C, -1)[:, :V]
    return -torch.log(-torch.log(((words >> 9).double() + 0.5) * 2.0 ** -23))


def _corrected64(z, prev, Ec, Wc, temperature):
    """Corrected logits of the block, each position conditioned on the token before it."""
    C, B, V = z.shape
    Wc, y = Wc.double(), prev.long()
    for i in range(B):
        z[:, i] += Ec[y].double() @ Wc.T
        score = z[:, i] if temperature == 0 else z[:, i] / temperature + _gumbel64(C, V, i, 3)
        y = score.float().argmax(-1)
    return z


def exact(case, seed):
    x, s, kind = _inputs(case, seed), _shape(case), case["kind"]
    if kind == "linear":
        w, a = x["w"], x["x"].double()
        return torch.cat([a @ w[n:n + 16384].double().T for n in range(0, w.shape[0], 16384)], 1)
    if kind == "verify":
        return None                                                  # whole numbers only
    if kind == "sample":
        return {"tokens": None, "logits": _corrected64(x["z"].double(), x["prev"], x["Ec"], x["Wc"], case["temperature"])}
    if kind == "fold":
        return {**_fold64(s, x["G"], x["state"], x["k"], x["v"], x["h"], x["acc"]), "t": None}
    if kind == "prefill":
        empty = {n: torch.zeros(sh, device=DEV) for n, sh, _ in _parts(s)}
        empty["eta"] -= math.inf
        acc = torch.tensor([case["t"]])
        return {**_fold64(s, x["G"], empty, x["k"][None], x["v"][None], x["h"][None], acc), "t": None}
    w, acc = x["w"], x["acc"]
    f = _fold64(s, w["G"], x["state"], x["k"], x["v"], x["h"], acc)
    z = _base64(s, w, f, x["state"]["t"] + acc, x["block"])
    return {"tokens": None, "logits": _corrected64(z, x["block"][:, 0], w["Ec"], w["Wc"], case["temperature"])}

"""Timed cases of the framework's public entry points.

Every case is work that a program around this library has it do: a draft-and-verify step
(`Context.compress`, then `Context.verify` with the fused draw), verification of target rows that
arrive in pieces (`verify_range`), the stand-alone draw (`residual_sample`), the exchange in the
other direction (`target_topk` on the verifier, `edge_resample` on the drafter) and the wire codec
of the sparse rows.  Outputs are written into tensors that the program keeps, where the entry point
takes them.

Inputs follow the recipe of `gen/` with one change that makes them quick to produce: the Zipf rank
of an entry is drawn uniformly from 1 .. V instead of being its place in a permutation.
"""
import torch

import paper_2603_19133_b200 as ps

# The smallest and the largest vocabulary, batch, draft length and sparse row of the drawn cases.
V_RANGE, B_RANGE, G_RANGE, K_RANGE = (8000, 262144), (1, 512), (1, 10), (1, 1024)
# a drawn case reads at most this much (the largest listed case)
MOST_BYTES = 512 * (8 + 9) * 262144 * 2


def listed():
    def case(name, kind, B, G, V, dtype, k, top_p=1.0):
        return {"name": name, "kind": kind, "B": B, "G": G, "V": V, "dtype": dtype, "k": k, "top_p": top_p}

    return [
        # one interactive sequence with a small vocabulary: launches and latency
        case("step_1x4_v32000_f32_k32", "step", 1, 4, 32000, "f32", 32),
        # a small serving batch, nucleus truncation capped at 64 entries
        case("step_8x5_v128256_bf16_p95_k64", "step", 8, 5, 128256, "bf16", 64, 0.95),
        # an ordinary batch, plain top-k
        case("step_64x8_v151936_bf16_k128", "step", 64, 8, 151936, "bf16", 128),
        # a full batch of concurrent sequences, nucleus truncation capped at 256 (the benchmark's workload)
        case("step_256x6_v128256_bf16_p90_k256", "step", 256, 6, 128256, "bf16", 256, 0.9),
        # the ends of the bandwidth sweep: the largest vocabulary with the widest rows, the smallest with narrow ones
        case("step_512x8_v262144_bf16_k1024", "step", 512, 8, 262144, "bf16", 1024),
        case("step_512x8_v32000_bf16_k8", "step", 512, 8, 32000, "bf16", 8),
        # a model head that leaves fp32 logits
        case("step_48x5_v128256_f32_p95_k64", "step", 48, 5, 128256, "f32", 64, 0.95),
        # an odd vocabulary without padding: rows start at any 2-byte boundary
        case("step_24x4_v50381_bf16_p90_k50", "step", 24, 4, 50381, "bf16", 50, 0.9),
        # target rows that arrive three at a time, drafts of unequal length
        case("range_64x8_v151936_bf16_k128", "range", 64, 8, 151936, "bf16", 128),
        # the draw by itself, at given positions, from target rows whose verification was done elsewhere
        case("residual_32x5_v128256_bf16_k64", "residual", 32, 5, 128256, "bf16", 64, 0.95),
        # verifier sends the ten largest components of the rejected row, drafter resamples
        case("paper_256x6_v128256_bf16_k10", "paper", 256, 6, 128256, "bf16", 10),
        # the sparse rows of a full batch to a message and back
        case("wire_256x6_k256", "wire", 256, 6, 128256, "bf16", 256, 0.9),
    ]


def draw(rng):
    """One more case: mostly whole steps, now and then one of the other calls."""
    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    while True:
        V = log_int(*V_RANGE)
        shape = rng.random()
        if shape < 0.7:
            V -= V % 64             # a padded vocabulary; the others stay as they fall, odd ones included
        case = {
            "kind": rng.choice(["step"] * 5 + ["range", "residual", "paper", "wire"]),
            "B": log_int(*B_RANGE), "G": rng.randint(*G_RANGE), "V": V,
            "dtype": rng.choice(["bf16", "bf16", "f32"]), "k": log_int(*K_RANGE),
            "top_p": rng.choice([1.0, round(rng.uniform(0.8, 0.99), 3)]),
        }
        size = 2 if case["dtype"] == "bf16" else 4
        if case["B"] * (2 * case["G"] + 1) * V * size <= MOST_BYTES:
            return case


def _logits(case, gen, want_draft, want_target):
    """Draft [B, G, V] and target [B, G+1, V] logits: base = -1.1 ln(rank) + 1.5 N(0,1) is the draft,
    rho * base + sqrt(1 - rho^2) * 1.5 N(0,1) the target, rho ~ U(0.5, 0.95) per sequence."""
    B, G, V = case["B"], case["G"], case["V"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    draft = torch.empty((B, G, V), dtype=dt, device="cuda") if want_draft else None
    target = torch.empty((B, G + 1, V), dtype=dt, device="cuda") if want_target else None
    rho = 0.5 + 0.45 * torch.rand((B, 1, 1), generator=gen, device="cuda")
    block = max(1, (1 << 27) // ((G + 1) * V))
    for b0 in range(0, B, block):
        n = min(B, b0 + block) - b0
        base = torch.rand((n, G + 1, V), generator=gen, device="cuda")
        base.mul_(V).floor_().add_(1.0).log_().mul_(-1.1)
        noise = torch.randn((n, G + 1, V), generator=gen, device="cuda")
        base.add_(noise, alpha=1.5)
        if want_draft:
            draft[b0:b0 + n] = base[:, :G]
        if want_target:
            noise = torch.randn((n, G + 1, V), generator=gen, device="cuda")
            r = rho[b0:b0 + n]
            target[b0:b0 + n] = base.mul_(r).add_(noise.mul_(torch.sqrt(1.0 - r * r) * 1.5))
    return draft, target


def _wire_rows(case, gen):
    """Sparse rows as nucleus truncation leaves them: counts from 1 to K, probabilities in falling order."""
    R, K = case["B"] * case["G"], case["k"]
    count = torch.randint(1, K + 1, (R,), generator=gen, device="cuda", dtype=torch.int32)
    live = torch.arange(K, device="cuda") < count[:, None]
    idx = torch.randint(0, case["V"], (R, K), generator=gen, device="cuda", dtype=torch.int32)
    prob = torch.rand((R, K), generator=gen, device="cuda").pow_(4).sort(dim=1, descending=True).values
    prob = torch.where(live, prob, torch.zeros_like(prob))
    prob /= prob.sum(dim=1, keepdim=True)
    return torch.where(live, idx, torch.full_like(idx, -1)), prob.contiguous(), count


def prepare(case, seed):
    B, G, V, K = case["B"], case["G"], case["V"], case["k"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    i32, f32 = torch.int32, torch.float32
    st = {"case": dict(case), "ctx": ps.Context(B, G, V, K)}

    def empty(shape, dtype):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    def uniform(*shape):
        return torch.rand(shape, generator=gen, device="cuda").clamp_(max=1.0 - 2.0 ** -24)

    if case["kind"] == "wire":
        R = B * G
        st["rows"] = _wire_rows(case, gen)
        st["buf"] = empty((ps.wire_bytes(R, R * K),), torch.uint8)
        st["bytes"] = empty((1,), torch.int64)
        st["out"] = (empty((R, K), i32), empty((R, K), f32), empty((R,), i32))
        return st

    st["draft"], st["target"] = _logits(case, gen, True, True)
    st["temperature"] = 0.5 + 0.7 * torch.rand((B,), generator=gen, device="cuda")
    st["u_draft"], st["u_accept"], st["u_resample"] = uniform(B, G), uniform(B, G), uniform(B, 2)
    st["sparse"] = (empty((B, G, K), i32), empty((B, G, K), f32), empty((B, G), i32), empty((B, G), i32))
    st["verdict"] = {"accept_len": empty((B,), i32), "p_draft": empty((B, G), f32), "resid_mass": empty((B, G), f32),
                     "borderline_count": empty((1,), i32), "token": empty((B,), i32)}
    if case["kind"] in ("range", "residual"):
        # the drafter's share is done by the time the target rows are there
        st["ctx"].compress(st["draft"], st["temperature"], K, case["top_p"], K, st["u_draft"], out=st["sparse"])
        st["draft"] = None
    if case["kind"] == "range":
        st["gamma"] = torch.randint(max(1, G // 2), G + 1, (B,), generator=gen, device="cuda", dtype=i32)
        st["verdict"]["state"] = empty((B,), i32)
    if case["kind"] in ("residual", "paper"):
        rows = G + 1 if case["kind"] == "residual" else G
        st["pos"] = torch.randint(0, rows, (B,), generator=gen, device="cuda", dtype=i32)
    if case["kind"] == "paper":
        st["top"] = (empty((B, K), i32), empty((B, K), f32), empty((B,), i32))
        st["drawn"] = (empty((B,), i32), empty((B,), f32))
        st["u"] = uniform(B)
    return st


def _windows(G):
    return [(r0, min(G + 1, r0 + 3)) for r0 in range(0, G + 1, 3)]


def run(st):
    case, ctx = st["case"], st["ctx"]
    if case["kind"] == "wire":
        buf, nbytes = ctx.wire_pack(*st["rows"], buf=st["buf"], bytes_out=st["bytes"])
        back = ctx.wire_unpack(buf, buf.numel(), case["B"] * case["G"], case["k"], out=st["out"])
        return [buf, nbytes, *back]
    T = st["temperature"]
    if case["kind"] == "step":
        idx, prob, count, tok = ctx.compress(st["draft"], T, case["k"], case["top_p"], case["k"], st["u_draft"], out=st["sparse"])
        v = ctx.verify(st["target"], T, tok, idx, prob, count, st["u_accept"], st["u_resample"], out=st["verdict"])
        return {"sparse": [idx, prob, count, tok], "verdict": v}
    idx, prob, count, tok = st["sparse"]
    if case["kind"] == "range":
        v, state = st["verdict"], None
        for r0, r1 in _windows(case["G"]):
            v = ctx.verify_range(st["target"], T, st["gamma"], r0, r1, state, tok, idx, prob, count, st["u_accept"],
                                 st["u_resample"], out=v)
            state = v["state"]
        return v
    if case["kind"] == "residual":
        token, mass = ctx.residual_sample(st["target"], T, st["pos"], idx, prob, count, st["u_resample"])
        return [token, mass]
    top = ctx.target_topk(st["target"], T, st["pos"], case["k"], out=st["top"])
    token, mass = ctx.edge_resample(st["draft"], T, st["pos"], *top, st["u"], out=st["drawn"])
    return {"top": list(top), "token": token, "mass": mass}


def work(case):
    """Logit rows that have to be read, sparse rows (8 bytes an entry) and per-position values; about
    three operations (scale, exponential, sum) on each logit."""
    B, G, V, K = case["B"], case["G"], case["V"], case["k"]
    size = 2 if case["dtype"] == "bf16" else 4
    sparse = B * G * (8 * K + 8)
    if case["kind"] == "wire":
        half = B * G * (K + 1) // 2                     # counts are uniform from 1 to K
        return {"bytes": 2 * (8 * half + 2 * B * G) + 8 * half + 8 * B * G * K, "flops": 0}
    if case["kind"] == "step":
        rows, extra = B * (2 * G + 1), 2 * sparse + B * G * 24
    elif case["kind"] == "range":
        # about every second sequence is decided by each window that it meets
        rows = sum(int(B * (r1 - r0) * 0.5 ** i) for i, (r0, r1) in enumerate(_windows(G)))
        extra = sparse + B * G * 12
    elif case["kind"] == "residual":
        rows, extra = B, B * (8 * K + 24)
    else:
        rows, extra = 2 * B, 2 * B * (8 * K + 16)
    return {"bytes": rows * V * size + extra, "flops": 3 * rows * V}


def tolerance(case):
    """Indices, counts, tokens and accept lengths are exact (decisions that fp32 sums cannot take are
    re-taken in double precision), and so is the codec.  Probabilities and residual masses carry the
    relative error of a normaliser summed in fp32 from the hardware exponential: against softmax in
    64 bits at most 1.2e-7 in the 2-norm and 3.4e-7 at the worst value over the listed cases; four times that."""
    if case["kind"] == "wire":
        return "exact"
    return {"rel": 5e-7, "max": 1.5e-6}


def _softmax(logits, T):
    """Rows [R, V] at their temperatures [R], in 64 bits."""
    return torch.softmax(logits.double() / T.double()[:, None], dim=1)


def _row_blocks(R, V):
    n = max(1, (1 << 26) // V)
    return [(i, min(R, i + n)) for i in range(0, R, n)]


def _pick(weight, u):
    """First entry at which the running sum of each row's weights exceeds u times its total."""
    run = weight.cumsum(1)
    return (run <= u.double()[:, None] * run[:, -1:]).sum(1).clamp_(max=weight.shape[1] - 1)


def _exact_compress(logits, T, K, top_p, u):
    """[R, V] rows: the K largest logits (ties: lower index first), the nucleus cut, the draw."""
    R, V = logits.shape
    n = min(K, V)
    idx = torch.full((R, K), -1, dtype=torch.int64, device=logits.device)
    prob = torch.zeros((R, K), dtype=torch.float64, device=logits.device)
    count = torch.empty((R,), dtype=torch.int64, device=logits.device)
    tok = torch.empty_like(count)
    for a, b in _row_blocks(R, V):
        p = _softmax(logits[a:b], T[a:b])
        order = logits[a:b].sort(dim=1, descending=True, stable=True).indices[:, :n]
        w = p.gather(1, order)
        m = (w.cumsum(1) < top_p).sum(1).add_(1).clamp_(max=n) if top_p < 1.0 else torch.full_like(count[a:b], n)
        live = torch.arange(n, device=w.device) < m[:, None]
        q = torch.where(live, w, torch.zeros_like(w))
        q /= q.sum(1, keepdim=True)
        idx[a:b, :n] = torch.where(live, order, torch.full_like(order, -1))
        prob[a:b, :n], count[a:b] = q, m
        if u is not None:
            tok[a:b] = order.gather(1, _pick(q, u[a:b])[:, None])[:, 0]
    return idx, prob, count, tok


def _exact_verify(st, idx, prob, tok):
    """p(x), the residual mass and the accept test of every draft position."""
    B, G, K = idx.shape
    V = st["target"].shape[2]
    logits = st["target"][:, :G].reshape(B * G, V)
    T = st["temperature"].repeat_interleave(G)
    idx, q, tok = idx.reshape(B * G, K), prob.reshape(B * G, K).double(), tok.reshape(B * G, 1)
    px, mass = (torch.empty((B * G,), dtype=torch.float64, device=q.device) for _ in range(2))
    for a, b in _row_blocks(B * G, V):
        p = _softmax(logits[a:b], T[a:b])
        px[a:b] = p.gather(1, tok[a:b].long())[:, 0]
        at = idx[a:b].clamp(min=0).long()
        mass[a:b] = p.scatter_add_(1, at, -q[a:b]).clamp_(min=0.0).sum(1)       # (an empty slot has q = 0)
    qx = torch.where(idx == tok, q, torch.zeros_like(q)).sum(1)
    accept = (qx <= 0) | (st["u_accept"].reshape(-1).double() < (px / qx).clamp(max=1.0))
    return px.reshape(B, G), mass.reshape(B, G), accept.reshape(B, G)


def exact(case, seed):
    """What `run` returns, in 64 bits from torch.  The drawn tokens of the two-level sampler and the
    count of borderline tests are left out; the codec's bytes are no computed numbers."""
    if case["kind"] == "wire":
        return None
    B, G, K = case["B"], case["G"], case["k"]
    st = prepare(case, seed)
    T = st["temperature"]
    seq = torch.arange(B, device=T.device)
    if case["kind"] == "step":
        R = B * G
        idx, prob, count, tok = _exact_compress(st["draft"].reshape(R, -1), T.repeat_interleave(G), K, case["top_p"],
                                                st["u_draft"].reshape(-1))
        # the rows are stored in 32 bits and verified as they are stored
        px, mass, accept = _exact_verify(st, idx.reshape(B, G, K), prob.float().reshape(B, G, K), tok)
        length = accept.long().cumprod(1).sum(1)
        return {"sparse": [idx.reshape(B, G, K), prob.reshape(B, G, K), count.reshape(B, G), tok.reshape(B, G)],
                "verdict": {"accept_len": length, "p_draft": px, "resid_mass": mass, "borderline_count": None, "token": None}}
    if case["kind"] == "range":
        idx, prob, count, tok = st["sparse"]
        px, mass, accept = _exact_verify(st, idx, prob, tok)
        gamma = st["gamma"].long()
        at = torch.arange(G, device=T.device)
        drafted = at < gamma[:, None]
        length = (accept & drafted).long().cumprod(1).sum(1)
        last = torch.zeros_like(length)         # first row after the window that decides the sequence
        for r0, r1 in _windows(G):
            last = torch.where((length >= r0) & (length < r1), torch.full_like(last, r1), last)
        seen = drafted & (at < last[:, None])
        return {"accept_len": length, "p_draft": px * seen, "resid_mass": mass * seen, "borderline_count": None,
                "token": None, "state": torch.zeros_like(length)}
    pos = st["pos"].long()
    p = _softmax(st["target"][seq, pos], T)
    if case["kind"] == "residual":
        idx, prob = st["sparse"][0], st["sparse"][1]
        row = pos.clamp(max=G - 1)
        q = prob[seq, row].double() * (pos < G)[:, None]
        return [None, p.scatter_add_(1, idx[seq, row].clamp(min=0).long(), -q).clamp_(min=0.0).sum(1)]
    idx, _, count, _ = _exact_compress(st["target"][seq, pos], T, K, 1.0, None)
    live = idx >= 0
    top = torch.where(live, p.gather(1, idx.clamp(min=0)), torch.zeros(1, dtype=p.dtype, device=p.device))
    sent = top.float().double()                 # the message carries 32 bits
    own = _softmax(st["draft"][seq, pos], T).gather(1, idx.clamp(min=0))
    left = torch.where(live, (sent - own).clamp(min=0.0), torch.zeros_like(own))
    return {"top": [idx, top, count], "token": None, "mass": left.sum(1)}

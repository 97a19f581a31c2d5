"""What the Python calls refuse: every tensor argument of every call on the CPU, with another type, of another
shape and with gaps, and logits that are not [B, R, V], is a ValueError before anything is launched; the
same call with the argument as it should be still runs."""
import pytest
import torch

pytestmark = pytest.mark.gpu

B, G, V, K, R = 3, 2, 2000, 8, 6
I32, F32, U8, I64 = torch.int32, torch.float32, torch.uint8, torch.int64


def _z(dtype, *shape):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def _calls(ctx):
    """name -> (call of a dict of tensors, the tensors, those whose shape the call does not fix)."""
    T = torch.ones((B,), device="cuda")
    rows = dict(q_idx=_z(I32, B, G, K), q_prob=_z(F32, B, G, K), q_count=_z(I32, B, G))
    rows["q_idx"][:] = torch.arange(K, device="cuda", dtype=I32)
    rows["q_prob"][:] = 1.0 / K
    rows["q_count"][:] = K
    draft = torch.randn((B, G, V), device="cuda")
    target = torch.randn((B, G + 1, V), device="cuda")
    verdict = dict(accept_len=_z(I32, B), p_draft=_z(F32, B, G), resid_mass=_z(F32, B, G), borderline_count=_z(I32, 1),
                   token=_z(I32, B))
    tests = dict(draft_tok=_z(I32, B, G), **rows, u_accept=_z(F32, B, G), u_resample=_z(F32, B, 2))
    top = dict(p_idx=_z(I32, B, K), p_prob=_z(F32, B, K), p_count=_z(I32, B))
    top["p_idx"][:] = torch.arange(K, device="cuda", dtype=I32)
    top["p_prob"][:] = 0.1
    top["p_count"][:] = K

    def verify(a):
        return ctx.verify(a["logits"], a["T"], *(a[n] for n in tests), out={n: a[n] for n in verdict})

    def verify_range(a):
        return ctx.verify_range(a["logits"], a["T"], a["gamma"], 0, G + 1, a["state_in"], *(a[n] for n in tests),
                                out={n: a[n] for n in (*verdict, "state")})

    flat = {n: t.reshape(R, *t.shape[2:]) for n, t in rows.items()}
    message = _z(U8, 16 + 2 * R + 8 * R * K + 8)
    nbytes = _z(I64, 1)
    ctx.wire_pack(*flat.values(), buf=message, bytes_out=nbytes)
    size = int(nbytes.item())
    return {
        "compress": (lambda a: ctx.compress(a["logits"], a["T"], K, 1.0, K, a["u_draft"],
                                            out=(a["idx"], a["prob"], a["count"], a["tok"])),
                     dict(logits=draft, T=T, u_draft=_z(F32, B, G), idx=_z(I32, B, G, K), prob=_z(F32, B, G, K),
                          count=_z(I32, B, G), tok=_z(I32, B, G)), ()),
        "verify": (verify, dict(logits=target, T=T, **tests, **verdict), ()),
        "verify_range": (verify_range, dict(logits=target, T=T, gamma=_z(I32, B) + G, state_in=_z(I32, B) + 1, **tests,
                                            **verdict, state=_z(I32, B)), ()),
        "residual_sample": (lambda a: ctx.residual_sample(a["logits"], a["T"], a["pos"], a["q_idx"], a["q_prob"],
                                                          a["q_count"], a["u"]),
                            dict(logits=target, T=T, pos=_z(I32, B), **rows, u=_z(F32, B, 2)), tuple(rows)),
        "target_topk": (lambda a: ctx.target_topk(a["logits"], a["T"], a["pos"], K, out=(a["idx"], a["prob"], a["count"])),
                        dict(logits=target, T=T, pos=_z(I32, B), idx=_z(I32, B, K), prob=_z(F32, B, K), count=_z(I32, B)), ()),
        "edge_resample": (lambda a: ctx.edge_resample(a["logits"], a["T"], a["pos"], a["p_idx"], a["p_prob"], a["p_count"],
                                                      a["u"], out=(a["token"], a["mass"])),
                          dict(logits=draft, T=T, pos=_z(I32, B), **top, u=_z(F32, B), token=_z(I32, B), mass=_z(F32, B)), ()),
        "wire_pack": (lambda a: ctx.wire_pack(a["q_idx"], a["q_prob"], a["q_count"], buf=a["buf"], bytes_out=a["bytes"]),
                      dict(**flat, buf=message.clone(), bytes=_z(I64, 1)), ("q_idx", "q_prob", "q_count", "buf")),
        "wire_unpack": (lambda a: ctx.wire_unpack(a["buf"], size, R, K, out=(a["idx"], a["prob"], a["count"])),
                        dict(buf=message, idx=_z(I32, R, K), prob=_z(F32, R, K), count=_z(I32, R)), ("buf",)),
    }


@pytest.mark.parametrize("name", ["compress", "verify", "verify_range", "residual_sample", "target_topk", "edge_resample",
                                  "wire_pack", "wire_unpack"])
def test_every_argument_is_checked(name):
    import paper_2603_19133_b200 as ps
    ctx = ps.Context(B, G, V, K)
    try:
        call, args, free = _calls(ctx)[name]
        call(args)
        assert ctx.status(clear=True)[0] == 0
        for arg, good in args.items():
            bad = [good.cpu(), good.to(torch.float64 if good.is_floating_point() else torch.int16)]
            wide = torch.zeros((*good.shape, 2), dtype=good.dtype, device="cuda")[..., 0]
            wide.copy_(good)
            if wide.numel() > 1:
                bad.append(wide)                                # the right shape and type, every other element
            if arg not in free:
                bad.append(good[None])
                if arg != "logits":
                    bad.append(torch.cat([good, good]))
            for b in bad:
                with pytest.raises(ValueError):
                    call({**args, arg: b})
        call(args)
        assert ctx.status(clear=True)[0] == 0
    finally:
        ctx.close()


def test_logits_that_are_no_logits():
    # refused as such also where the call makes its own outputs from their shape
    import paper_2603_19133_b200 as ps
    ctx = ps.Context(B, G, V, K)
    try:
        calls = _calls(ctx)
        v, r = calls["verify"][1], calls["residual_sample"][1]
        tests = [v[n] for n in ("draft_tok", "q_idx", "q_prob", "q_count", "u_accept", "u_resample")]
        e = calls["edge_resample"][1]
        for shape in ((), (V,), (B, V), (B, G + 1, V, 1)):
            x = torch.zeros(shape, device="cuda")
            for f in (lambda: ctx.compress(x, v["T"], K, 1.0, K),
                      lambda: ctx.verify(x, v["T"], *tests),
                      lambda: ctx.verify_range(x, v["T"], None, 0, G + 1, None, *tests),
                      lambda: ctx.residual_sample(x, v["T"], r["pos"], r["q_idx"], r["q_prob"], r["q_count"], r["u"]),
                      lambda: ctx.target_topk(x, v["T"], r["pos"], K),
                      lambda: ctx.edge_resample(x, v["T"], r["pos"], e["p_idx"], e["p_prob"], e["p_count"], e["u"])):
                with pytest.raises(ValueError):
                    f()
    finally:
        ctx.close()

"""Rows at every offset from a 16-byte boundary through the staged kernels: compress, verify and the
stand-alone draw against the oracle (whole numbers bit-exact, the rest to 1e-5), with NaN around
every row so that a neighbour's entry that gets into a result shows."""
import numpy as np
import pytest
import torch

import gen
import oracle

pytestmark = pytest.mark.gpu


def _offset_copy(t, offset, gap):
    B, R, V = t.shape
    pitch = V + gap
    flat = torch.full((offset + B * R * pitch,), float("nan"), dtype=t.dtype, device=t.device)
    view = flat[offset:].view(B, R, pitch)[:, :, :V]
    view.copy_(t)
    return view


def _np(t):
    return t.float().cpu().numpy() if t.is_floating_point() else t.cpu().numpy()


@pytest.mark.parametrize("dtype,V,offset,gap,K,top_p", [
    ("bf16", 3, 5, 2, 2, 1.0),              # a row inside one granule
    ("bf16", 11, 6, 1, 4, 0.9),             # two granules, neither full
    ("bf16", 1024, 1, 7, 16, 1.0),          # one chunk and a granule of the next virtual one
    ("bf16", 1025, 7, 0, 16, 0.9),
    ("bf16", 8192, 7, 1, 64, 1.0),          # a full tile, shifted: the row's last entries lie in the tile behind it
    ("bf16", 8192, 1, 15, 64, 0.9),
    ("bf16", 8193, 0, 0, 200, 1.0),         # the offset changes from row to row
    ("bf16", 16384, 3, 0, 700, 0.95),
    ("bf16", 16377, 7, 16, 64, 1.0),        # offset and length make whole tiles
    ("bf16", 50381, 1, 0, 50, 0.9),
    ("bf16", 131073, 0, 0, 64, 0.95),       # few long rows, dealt in pieces
    ("f32", 5, 1, 0, 3, 1.0),
    ("f32", 1024, 3, 1, 16, 0.9),
    ("f32", 8192, 2, 0, 64, 1.0),
    ("f32", 16385, 1, 0, 128, 0.95),
    ("f32", 24575, 0, 0, 600, 1.0),
    ("f32", 98305, 3, 2, 40, 0.95),
])
def test_rows_at_any_offset(dtype, V, offset, gap, K, top_p):
    import paper_2603_19133_b200 as ps
    B, G = 5, 2
    w = gen.Workload("t", V=V, B=B, G=G, dtype=dtype, s=1.1, sigma_d=1.5, corr=0.8, sigma_t=1.0, T=None,
                     top_k=0 if top_p < 1.0 else K, top_p=top_p, k_max=K)
    inp = gen.make_inputs(w, seed=V + offset, device="cuda")
    dl, tl = (_offset_copy(inp[n], offset, gap) for n in ("draft_logits", "target_logits"))
    T, ua, ur = inp["temperature"], inp["u_accept"], inp["u_resample"]
    ctx = ps.Context(B, G, V, K)
    try:
        qi, qp, qc, tok = ctx.compress(dl, T, w.top_k, top_p, K, inp["u_draft"])
        g = ctx.verify(tl, T, tok, qi, qp, qc, ua, ur)
        pos = g["accept_len"].clone()
        tok2, mass = ctx.residual_sample(tl, T, pos, qi, qp, qc, ur)
        assert ctx.status(clear=True)[0] == 0
    finally:
        ctx.close()
    o_qi, o_qp, o_qc, o_tok = oracle.compress(_np(inp["draft_logits"]), _np(T), w.top_k, top_p, K, _np(inp["u_draft"]))
    for a, b in ((qi, o_qi), (qc, o_qc), (tok, o_tok)):
        assert np.array_equal(_np(a), b)
    np.testing.assert_allclose(_np(qp), o_qp, rtol=1e-5)
    o = oracle.verify(_np(inp["target_logits"]), _np(T), o_tok, o_qi, _np(qp), o_qc, _np(ua), _np(ur))
    assert np.array_equal(_np(g["accept_len"]), o["accept_len"]) and np.array_equal(_np(g["token"]), o["token"])
    assert int(g["borderline_count"].item()) == o["borderline_count"]
    np.testing.assert_allclose(_np(g["p_draft"]), o["p_draft"], rtol=1e-5)
    # (masses are differences from one of sums in double precision: 1e-12)
    np.testing.assert_allclose(_np(g["resid_mass"]), o["resid_mass"], rtol=1e-5, atol=1e-12)
    assert np.array_equal(_np(tok2), o["token"])

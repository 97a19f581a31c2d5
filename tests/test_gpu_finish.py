"""The counting sort of the compress finish: groups of 32 and of 256 threads, ties across the k-th
place up to and beyond the group's buffer, values beyond the last bin, rows put together from pieces.
Supports, counts and draws are bit-exact against the oracle, probabilities agree to 1e-5."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rows,V,k,above,ties,binades,redo", [
    (9, 16384, 1, 0, 5, 0, 0),               # one key kept of five equal ones; a warp per row, a part-filled CTA
    (5, 16384, 128, 127, 385, 3, 0),         # the largest k of a warp; ties that exactly fill its buffer (512)
    (5, 16384, 128, 127, 390, 3, 5),         # five more than the scratch area holds: the direct kernel
    (5, 16384, 129, 100, 412, 3, 0),         # the smallest k of a CTA
    (5, 16384, 128, 128, 0, 24, 0),          # 24 binades above the bound: most keys share the open last bin (4 binades)
    (4, 16384, 300, 290, 60, 24, 0),         # the same for a CTA (16 binades)
    (3, 65536, 1024, 1000, 1048, 6, 0),      # CTA buffer exactly full (2048)
    (3, 131072, 40, 30, 200, 3, 0),          # eight pieces per row, ties in all of them
])
def test_select_and_order(rows, V, k, above, ties, binades, redo, dtype):
    import paper_2603_19133_b200 as ps
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(rows * V + k + ties)
    dl = torch.rand((rows, 1, V), generator=g, device="cuda") * 4.0 - 6.0          # filler in [-6, -2)
    for r in range(rows):
        perm = torch.randperm(V, generator=g, device="cuda")
        step = torch.arange(above, device="cuda")
        dl[r, 0, perm[:above]] = 2.0 ** (1.0 + binades * (step + 1.0) / (above + 1.0))
        dl[r, 0, perm[above:above + ties]] = 0.5
    dl = dl.to(td)
    T = torch.full((rows,), 2.0 ** max(0, binades - 4), device="cuda")
    u = torch.rand((rows, 1), generator=g, device="cuda")
    ctx = ps.Context(rows, 1, V, k)
    try:
        got = [t.cpu().numpy() for t in ctx.compress(dl, T, k, 1.0, k, u)]
        assert ctx.counters(clear=True)[1] == redo
        assert ctx.status(clear=True)[0] == 0
    finally:
        ctx.close()
    want = oracle.compress(dl.float().cpu().numpy(), T.cpu().numpy(), k, 1.0, k, u.cpu().numpy(), nthreads=oracle.cores())
    for a, b in ((got[0], want[0]), (got[2], want[2]), (got[3], want[3])):
        assert np.array_equal(a, b)
    np.testing.assert_allclose(got[1], want[1], rtol=1e-5)


@pytest.mark.parametrize("top_p", [1.0, 0.9])
@pytest.mark.parametrize("rows,V,k,head,redo", [
    (460, 65536, 256, 1.0 / 8, False),       # the large logits spread over the row (whole rows and pieces)
    (5, 131072, 100, 0.6, False),            # six in ten of them in the first eighth
    (5, 65536, 256, 1.0, False),             # all of them in the first eighth, spread over it
    (5, 65536, 256, -1.0, True),             # all of them in 512 neighbouring entries: the bound rises past the k-th
])
def test_bound_ahead_of_the_rows_end(rows, V, k, head, redo, top_p):
    # where the k largest lie must not show in the result, only in whether the direct kernel is needed
    import paper_2603_19133_b200 as ps
    g = torch.Generator(device="cuda").manual_seed(rows + V + k)
    dl = torch.randn((rows, 1, V), generator=g, device="cuda").clamp_(max=3.9)
    n = 2 * k
    for r in range(rows):
        if head < 0:
            at = 1024 * (r % 3) + torch.randperm(n, generator=g, device="cuda")
        else:
            m = int(round(n * head))
            first = torch.randperm(V // 8, generator=g, device="cuda")[:m]
            rest = V // 8 + torch.randperm(V - V // 8, generator=g, device="cuda")[:n - m]
            at = torch.cat([first, rest])
        dl[r, 0, at] = 4.0 + 3.0 * torch.rand(n, generator=g, device="cuda")
    dl = dl.to(torch.bfloat16)
    T = torch.full((rows,), 0.8, device="cuda")
    u = torch.rand((rows, 1), generator=g, device="cuda")
    top_k = k if top_p >= 1.0 else 0
    ctx = ps.Context(rows, 1, V, k)
    try:
        got = [t.cpu().numpy() for t in ctx.compress(dl, T, top_k, top_p, k, u)]
        redone = ctx.counters(clear=True)[1]
        assert ctx.status(clear=True)[0] == 0
    finally:
        ctx.close()
    assert redone == (rows if redo else 0)
    want = oracle.compress(dl.float().cpu().numpy(), T.cpu().numpy(), top_k, top_p, k, u.cpu().numpy(), nthreads=oracle.cores())
    for a, b in ((got[0], want[0]), (got[2], want[2]), (got[3], want[3])):
        assert np.array_equal(a, b)
    np.testing.assert_allclose(got[1], want[1], rtol=1e-5)

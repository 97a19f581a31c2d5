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

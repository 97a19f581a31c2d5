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
@pytest.mark.parametrize("rows,V,k,head", [
    (460, 65536, 256, 1.0 / 8),              # the large logits spread over the row (whole rows and pieces)
    (5, 131072, 100, 0.6),                   # six in ten of them in the first eighth
    (5, 65536, 256, 1.0),                    # all of them in the first eighth, spread over it
    (5, 65536, 256, -1.0),                   # all of them in 512 neighbouring entries
])
def test_bound_ahead_of_the_rows_end(rows, V, k, head, top_p):
    # where the k largest lie must show neither in the result nor in whether the direct kernel is needed
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
    _check_compress(dl.to(torch.bfloat16), k, top_p, 0.8, g)


def _check_compress(dl, k, top_p, temperature, g, staged=True):
    """Against the oracle; `staged`: no row is handed to the direct kernel."""
    import paper_2603_19133_b200 as ps
    rows, _, V = dl.shape
    T = torch.full((rows,), temperature, device="cuda")
    u = torch.rand((rows, 1), generator=g, device="cuda")
    top_k = k if top_p >= 1.0 else 0
    ctx = ps.Context(rows, 1, V, k)
    try:
        got = [t.cpu().numpy() for t in ctx.compress(dl, T, top_k, top_p, k, u)]
        redone = ctx.counters(clear=True)[1]
        assert ctx.status(clear=True)[0] == 0
    finally:
        ctx.close()
    assert redone == 0 or not staged
    want = oracle.compress(dl.float().cpu().numpy(), T.cpu().numpy(), top_k, top_p, k, u.cpu().numpy(), nthreads=oracle.cores())
    for a, b in ((got[0], want[0]), (got[2], want[2]), (got[3], want[3])):
        assert np.array_equal(a, b)
    np.testing.assert_allclose(got[1], want[1], rtol=1e-5)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V,k,top_p", [(128256, 64, 0.95), (128256, 1024, 1.0), (262144, 256, 0.9), (32000, 8, 1.0),
                                       (32000, 256, 1.0), (17409, 500, 1.0), (50381, 512, 0.95)])
@pytest.mark.parametrize("order", ["quarter", "half", "rank", "mixed", "reversed", "unused", "block"])
def test_vocabularies_with_an_order(V, k, top_p, order, dtype):
    # a vocabulary numbered by frequency, with an unused end, with a block of one language: the rows are as
    # right as any, and (but for logits that follow the numbers altogether) none of them is read a
    # second time by the direct kernel
    g = torch.Generator(device="cuda").manual_seed(V + k)
    rows = 6
    ids = torch.arange(V, device="cuda").float()
    noise = 1.5 * torch.randn((rows, V), generator=g, device="cuda")
    free = -1.1 * torch.log(torch.floor(torch.rand((rows, V), generator=g, device="cuda") * V) + 1.0)
    x = free + noise
    if order == "rank":
        x = noise - 1.1 * torch.log(ids + 1.0)
    elif order == "mixed":
        x = noise + 0.5 * free - 0.55 * torch.log(ids + 1.0)
    elif order == "reversed":
        x = noise - 1.1 * torch.log(V - ids)
    elif order == "unused":
        x[:, V * 7 // 8:] = -30.0
    elif order == "block":
        x[:, V // 4:V * 43 // 100] += 2.0
    else:
        # a quarter or a half of the k largest among the ids below 1024
        m = max(1, int(k * (0.25 if order == "quarter" else 0.5)))
        at = torch.rand((rows, 1024), generator=g, device="cuda").argsort(dim=1)[:, :m]
        kth = torch.topk(x, k - m + 1, dim=1).values[:, -1:]
        top = x.amax(dim=1, keepdim=True)
        x.scatter_(1, at, kth + 0.02 + 0.9 * (top - kth) * torch.rand((rows, m), generator=g, device="cuda"))
    _check_compress(x[:, None].to(torch.bfloat16 if dtype == "bf16" else torch.float32), k, top_p, 0.9, g,
                    staged=order not in ("rank", "reversed"))


@pytest.mark.parametrize("dtype,rows,V,k,offset", [
    ("bf16", 9, 32768, 1024, 100.0),         # several hundred keys of one code, for a CTA
    ("f32", 9, 32768, 1024, 100.0),
    ("f32", 5, 131072, 1024, 100.0),         # the same put together from pieces
    ("f32", 9, 32768, 300, 30.0),            # stretches below and above the limit in one row
    ("bf16", 9, 16384, 128, 100.0),          # for a warp
    ("f32", 9, 16384, 128, 100.0),
    ("f32", 9, 16384, 100, 100.0),
])
def test_many_keys_of_one_code(dtype, rows, V, k, offset):
    # a common offset leaves few 16-bit codes to the k largest: a network orders them instead of the counts
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = 2.0 * torch.randn((rows, 1, V), generator=g, device="cuda") + offset
    _check_compress(x.to(torch.bfloat16 if dtype == "bf16" else torch.float32), k, 1.0, 0.9, g, staged=k > 128)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("k,top_p", [(64, 1.0), (64, 0.9), (300, 0.9)])
@pytest.mark.parametrize("more", [0, 1])
def test_rows_to_read_again_among_few_and_many(more, k, top_p, dtype):
    # as many rows as are finished by a CTA that reads a row again itself (two per SM), and one more: then by
    # a warp (k = 64) or a CTA that lists such rows for another kernel.  Every ninth row is full of ties.
    rows, V = 2 * torch.cuda.get_device_properties(0).multi_processor_count + more, 16384
    g = torch.Generator(device="cuda").manual_seed(rows + k)
    x = 1.5 * torch.randn((rows, 1, V), generator=g, device="cuda")
    x[::9, :, :V // 2] = 3.0
    _check_compress(x.to(torch.bfloat16 if dtype == "bf16" else torch.float32), k, top_p, 0.8, g, staged=False)


@pytest.mark.parametrize("rows,V", [(400, 16384), (24, 16384), (24, 4096)])
def test_a_captured_call_is_replayed_alone(rows, V):
    # rows of equal logits whose cut falls on an entry's edge: each is read again by the direct kernel and takes
    # the double-precision cut.  A replay has no other call before it that would clear the lists.
    import paper_2603_19133_b200 as ps
    k, keep = 64, 40
    x = torch.zeros((rows, 1, V), dtype=torch.bfloat16, device="cuda")
    T = torch.ones((rows,), device="cuda")
    u = torch.rand((rows, 1), device="cuda")
    i32 = torch.int32
    out = (torch.empty((rows, 1, k), dtype=i32, device="cuda"), torch.empty((rows, 1, k), device="cuda"),
           torch.empty((rows, 1), dtype=i32, device="cuda"), torch.empty((rows, 1), dtype=i32, device="cuda"))
    ctx = ps.Context(rows, 1, V, k)
    try:
        ctx.compress(x, T, 0, keep / V, k, u, out=out)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ctx.compress(x, T, 0, keep / V, k, u, out=out)
        ctx.counters(clear=True)
        for n in range(1, 4):
            graph.replay()
            assert ctx.counters()[0] == n * rows
            assert (out[2] == keep).all() and (out[0][:, 0, :keep] == torch.arange(keep, dtype=i32, device="cuda")).all()
        assert ctx.status()[0] == 0
        del graph
    finally:
        ctx.close()


@pytest.mark.parametrize("V", [4096, 16384])
@pytest.mark.parametrize("order", ["eager capture eager", "eager replay eager", "replay replay eager replay"])
def test_captured_calls_between_others(order, V):
    # every row takes the double-precision cut, so each call leaves a full queue; the last call has fewer rows and
    # another vocabulary, for which a row number or a ticket left behind would lie outside its logits
    import paper_2603_19133_b200 as ps
    rows, k, keep, i32 = 24, 64, 40, torch.int32

    def inputs(n, v):
        out = (torch.empty((n, 1, k), dtype=i32, device="cuda"), torch.empty((n, 1, k), device="cuda"),
               torch.empty((n, 1), dtype=i32, device="cuda"), torch.empty((n, 1), dtype=i32, device="cuda"))
        return torch.zeros((n, 1, v), dtype=torch.bfloat16, device="cuda"), torch.ones((n,), device="cuda"), torch.rand((n, 1), device="cuda"), out

    def call(x, T, u, out):
        ctx.compress(x, T, 0, keep / x.shape[2], k, u, out=out)

    def check(x, T, u, out):
        assert (out[2] == keep).all() and (out[0][:, 0, :keep] == torch.arange(keep, dtype=i32, device="cuda")).all()
        for t in out[:3]:
            t.fill_(-7)

    ctx = ps.Context(rows, 1, V, k)
    try:
        full, small = inputs(rows, V), inputs(5, V * 5 // 8)      # (keep / V is exact in both)
        call(*full)
        check(*full)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call(*full)
        ctx.counters(clear=True)
        done = 0
        for step in order.split()[1:]:
            if step == "capture":
                continue
            if step == "replay":
                graph.replay()
                done += rows
                assert ctx.counters()[0] == done
                check(*full)
            else:
                call(*small)
                done += 5
                assert ctx.counters()[0] == done
                check(*small)
        call(*small)
        assert ctx.counters()[0] == done + 5
        check(*small)
        assert ctx.status()[0] == 0
        del graph
    finally:
        ctx.close()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V,k,share", [(16384, 1024, 1 / 3), (12000, 800, 1 / 2), (12000, 1024, 1 / 4)])
def test_crowded_place_in_rows_of_two_tiles(V, k, share, dtype):
    # more than 512 wanted of a row that has no more than two tiles, a share of them among the ids below 1024: a warp's
    # region holds its chunk's part of them, so that no row is read again
    rows, m = 60, int(k * share)
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = 1.5 * torch.randn((rows, V), generator=g, device="cuda") - 1.1 * torch.log(torch.floor(torch.rand((rows, V), generator=g, device="cuda") * V) + 1.0)
    at = torch.rand((rows, 1024), generator=g, device="cuda").argsort(dim=1)[:, :m]
    kth = torch.topk(x, k - m + 1, dim=1).values[:, -1:]
    x.scatter_(1, at, kth + 0.02 + 0.9 * (x.amax(dim=1, keepdim=True) - kth) * torch.rand((rows, m), generator=g, device="cuda"))
    _check_compress(x[:, None].to(torch.bfloat16 if dtype == "bf16" else torch.float32), k, 1.0, 0.9, g)

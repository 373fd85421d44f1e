"""Calls back to back without a synchronisation, sharing workspaces and outputs, on one stream and on two, directly and from a
captured graph: a kernel that starts while its predecessor runs must not read or overwrite anything early.  With four heads every
CTA has one tile of work; with 130 there are more tiles than SMs, and CTAs take those of others that have not started yet."""
import pytest

pytestmark = pytest.mark.gpu
HEADS = [4, 130]


def _state(seed, dtype, n, d, h=4):
    import torch
    g = torch.Generator("cuda").manual_seed(seed)
    return [torch.randn(1, h, n, d, device="cuda", generator=g).to(dtype) for _ in range(4)]


def _step(attn, x, out, ws, mask, cfg):
    q, k, v, do = x
    attn.attn_fwd(q, k, v, out[0], out[1], mask=mask, cfg=cfg, workspace=ws)
    attn.attn_bwd(q, k, v, out[0], do, out[1], *out[2:], mask=mask, cfg=cfg, workspace=ws)


@pytest.mark.parametrize("dtype,n,d,det", [("f32", 100, 64, 0), ("bf16", 320, 64, 1), ("bf16", 320, 128, 1), ("bf16", 331, 64, 1)])
@pytest.mark.parametrize("how", ["stream", "two_streams", "graph"])
@pytest.mark.parametrize("heads", HEADS)
def test_back_to_back_steps_equal_separate_ones(dtype, n, d, det, how, heads):
    import torch
    import paper_2410_09397_b200 as attn
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    cfg, mask = attn.Cfg(deterministic=det), attn.Mask(kind=attn.ATTN_MASK_CAUSAL)      # repeatable: compared bit for bit
    code = attn.ATTN_F32 if dtype == "f32" else attn.ATTN_BF16
    size = attn.attn_bwd_workspace_bytes(n, d, heads, 1, mask, code, cfg)
    xs = [_state(90 + i, dt, n, d, heads) for i in range(2)]

    def buffers():
        like = xs[0][0]
        return ([torch.zeros_like(like), torch.zeros(1, heads, n, device="cuda")] + [torch.zeros_like(like) for _ in range(3)],
                torch.full((size,), 255, dtype=torch.uint8, device="cuda"))     # garbage: the status word too
    want = []
    for x in xs:
        out, ws = buffers()
        _step(attn, x, out, ws, mask, cfg)
        torch.cuda.synchronize()
        want.append(out)
    got = []
    if how == "two_streams":
        streams = [torch.cuda.Stream() for _ in xs]
        bufs = [buffers() for _ in xs]
        torch.cuda.synchronize()
        for _ in range(5):
            for s, x, (out, ws) in zip(streams, xs, bufs):
                with torch.cuda.stream(s):
                    _step(attn, x, out, ws, mask, cfg)
        torch.cuda.synchronize()
        got = [b[0] for b in bufs]
        spaces = [b[1] for b in bufs]
    else:
        out, ws = buffers()
        spaces = [ws]
        kept = [[torch.empty_like(t) for t in out] for _ in xs]

        def run():
            for x, to in zip(xs, kept):       # the same outputs and workspace, copied out between the steps
                _step(attn, x, out, ws, mask, cfg)
                for a, b in zip(to, out):
                    a.copy_(b)
        if how == "graph":
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                run()
            for _ in range(3):
                graph.replay()
        else:
            for _ in range(3):
                run()
        torch.cuda.synchronize()
        got = kept
    assert all(attn.attn_workspace_status(ws) == attn.ATTN_OK for ws in spaces)
    for g, w in zip(got, want):
        assert all(torch.equal(a, b) for a, b in zip(g, w))


def _mask(attn, kind, n):
    import torch
    g = torch.Generator("cuda").manual_seed(89)
    if kind == "element":
        words = (n + 31) // 32
        bits = torch.randint(-2 ** 31, 2 ** 31, (1, n, words), dtype=torch.int32, device="cuda", generator=g)
        return attn.Mask(kind=attn.ATTN_MASK_ELEMENT, block_mask=bits)
    if kind == "fine":
        nb = (n + 63) // 64
        keep = torch.rand(1, nb, nb, device="cuda", generator=g) < 0.5
        keep[0].fill_diagonal_(True)
        return attn.Mask(kind=attn.ATTN_MASK_BLOCK_SPARSE, block=64, block_mask=keep.to(torch.uint8))
    return attn.Mask(kind=attn.ATTN_MASK_CAUSAL)


def _close(got, want):
    """Sums of fp32 atomics in another order (1e-6 apart), rounded to bf16: entries on the other side of a rounding boundary
    are 2^-8 apart, and 2e-3 allows one entry in four of them."""
    return (got.double() - want.double()).norm() <= 2e-3 * want.double().norm()


# (name, n, d, mask, cfg): every kernel of the default path, whose dQ is cleared by the pass before the backward, added to in
# atomics and converted by the pass after it; lists and bitmaps of masks in the workspace; the two-term kernels; the
# materialised path, whose own kernels are launched the ordinary way behind a pass that lets its successor start early
ROUTES = [("fused", 320, 64, "causal", {}), ("fused", 320, 128, "causal", {}), ("fused64", 320, 128, "causal", {"tile_q": 64}),
          ("wide", 320, 256, "causal", {}), ("two_terms", 331, 64, "causal", {}), ("two_terms", 331, 128, "causal", {}),
          ("element", 328, 64, "element", {}), ("element", 328, 128, "element", {}), ("fine", 328, 128, "fine", {}),
          ("two_terms_element", 331, 128, "element", {}), ("materialised", 320, 256, "causal", {"materialised": True})]


@pytest.mark.parametrize("name,n,d,kind,options", ROUTES)
@pytest.mark.parametrize("how", ["stream", "two_streams", "graph"])
@pytest.mark.parametrize("heads", HEADS)
def test_default_routes_back_to_back_equal_separate_calls(name, n, d, kind, options, how, heads):
    """Two problems in turn on the same outputs and workspace.  O, LSE, dK and dV have a fixed order of summation and are compared
    bit for bit, dQ within its atomics (exactly where there are none)."""
    import torch
    import paper_2410_09397_b200 as attn
    if options.get("materialised"):
        cfg = attn.Cfg(algo=attn.ATTN_ALGO_MATERIALIZED)
    elif "tile_q" in options:
        cfg = attn.Cfg(algo=attn.ATTN_ALGO_FUSED, tile_q=options["tile_q"])
    else:
        cfg = attn.Cfg()
    mask = _mask(attn, kind, n)
    size = max(attn.attn_fwd_workspace_bytes(n, d, heads, 1, mask, attn.ATTN_BF16, cfg),
               attn.attn_bwd_workspace_bytes(n, d, heads, 1, mask, attn.ATTN_BF16, cfg))
    xs = [_state(90 + i, torch.bfloat16, n, d, heads) for i in range(2)]

    def buffers():
        like = xs[0][0]
        return ([torch.zeros_like(like), torch.zeros(1, heads, n, device="cuda")] + [torch.zeros_like(like) for _ in range(3)],
                torch.full((size,), 255, dtype=torch.uint8, device="cuda"))
    want = []
    for x in xs:
        out, ws = buffers()
        _step(attn, x, out, ws, mask, cfg)
        torch.cuda.synchronize()
        want.append(out)
    sides = 2 if how == "two_streams" else 1
    bufs = [buffers() for _ in range(sides)]
    kept = [[[torch.empty_like(t) for t in bufs[0][0]] for _ in xs] for _ in range(sides)]

    def run(side):
        out, ws = bufs[side]
        for x, to in zip(xs, kept[side]):
            _step(attn, x, out, ws, mask, cfg)
            for a, b in zip(to, out):
                a.copy_(b)
    torch.cuda.synchronize()
    if how == "graph":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(0)
        for _ in range(3):
            graph.replay()
    else:
        streams = [torch.cuda.Stream() for _ in range(sides)]
        for _ in range(3):
            for side, s in enumerate(streams):
                with torch.cuda.stream(s):
                    run(side)
    torch.cuda.synchronize()
    assert all(attn.attn_workspace_status(ws) == attn.ATTN_OK for _, ws in bufs)
    exact = "two_terms" in name or name == "materialised"
    for side in kept:
        for g, w in zip(side, want):
            for what, a, b in zip(("O", "LSE", "dQ", "dK", "dV"), g, w):
                assert torch.equal(a, b) if what != "dQ" or exact else _close(a, b), what


@pytest.mark.parametrize("d", [64, 256])
@pytest.mark.parametrize("how", ["stream", "two_streams", "graph"])
@pytest.mark.parametrize("h", HEADS)
def test_weights_steps_back_to_back_equal_separate_ones(d, how, h):
    """Projections, forward and weight gradients of two problems in turn; gX and gY hold garbage before every call."""
    import torch
    import paper_2410_09397_b200 as attn
    n, mask, cfg = 328, attn.Mask(kind=attn.ATTN_MASK_CAUSAL), attn.Cfg()
    size = max(256, attn.attn_fwd_workspace_bytes(n, d, h, 1, mask, attn.ATTN_BF16, cfg),
               attn.attn_weights_bwd_workspace_bytes(n, d, h, 1, mask, attn.ATTN_BF16, cfg))
    xs = [_state(190 + i, torch.bfloat16, n, d, h) for i in range(2)]
    g = torch.Generator("cuda").manual_seed(192)
    X, Y = ((torch.randn(h, d, d, device="cuda", generator=g) / d ** 0.5).bfloat16() for _ in range(2))

    def buffers():
        like = xs[0][0]
        return ([torch.zeros_like(like) for _ in range(3)] + [torch.zeros(1, h, n, device="cuda")] +
                [torch.empty(h, d, d, device="cuda") for _ in range(2)], torch.full((size,), 255, dtype=torch.uint8, device="cuda"))

    def step(x, out, ws):
        q, k, v, do = x
        S, H, O, L, gX, gY = out
        gX.fill_(float("nan"))
        gY.fill_(float("nan"))
        attn.attn_project(q, X, S, workspace=ws)
        attn.attn_project(v, Y, H, workspace=ws)
        attn.attn_fwd(S, k, H, O, L, mask=mask, cfg=cfg, workspace=ws)
        attn.attn_weights_bwd(q, k, v, S, H, O, do, L, h, gX, gY, mask=mask, cfg=cfg, workspace=ws)
    want = []
    for x in xs:
        out, ws = buffers()
        step(x, out, ws)
        torch.cuda.synchronize()
        want.append(out)
    sides = 2 if how == "two_streams" else 1
    bufs = [buffers() for _ in range(sides)]
    kept = [[[torch.empty_like(t) for t in bufs[0][0]] for _ in xs] for _ in range(sides)]

    def run(side):
        for x, to in zip(xs, kept[side]):
            step(x, *bufs[side])
            for a, b in zip(to, bufs[side][0]):
                a.copy_(b)
    torch.cuda.synchronize()
    if how == "graph":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(0)
        for _ in range(3):
            graph.replay()
    else:
        streams = [torch.cuda.Stream() for _ in range(sides)]
        for _ in range(3):
            for side, s in enumerate(streams):
                with torch.cuda.stream(s):
                    run(side)
    torch.cuda.synchronize()
    assert all(attn.attn_workspace_status(ws) == attn.ATTN_OK for _, ws in bufs)
    for side in kept:
        for got, w in zip(side, want):
            assert all(torch.equal(a, b) for a, b in zip(got[:4], w[:4]))
            assert all(_close(a, b) for a, b in zip(got[4:], w[4:]))

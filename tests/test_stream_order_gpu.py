"""The calls keep their stream's order although each may be set up while the
kernel before it runs: inputs written by the kernel just before a call, by
another stream joined with an event, and calls back to back on one context,
eagerly and in a captured graph."""
import numpy as np
import pytest
import torch

from paper_2608_28726_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_28726_gb300 import binding
    return binding


def _calls(B, ctx, x, ch, off, feat, hw, qw, w, out):
    """route, features + pooling, a decode step, the head and the quantile scorer, back to back"""
    score, ship, fl, agg, rec, top2, rf, hs, hsh, hf, qs, qsh, qf, qsum, ds, dsh, df, da = out
    n = x.size(0)
    B.pr_route(ctx, x, ch, off, w, 0.1, 0.5, score=score, ship=ship, req_flags=fl, agg=agg)
    B.pr_token_features(ctx, x, ch, 20, off, rec, top2, rf)
    B.pr_aggregate_score(ctx, rec, off, w, 0.1, 0.5, rf, agg, score, ship, fl)
    slot = torch.arange(n, dtype=torch.int32, device="cuda")
    eos = torch.ones(n, dtype=torch.uint8, device="cuda")
    B.pr_decode_step(ctx, x, slot, ch, eos, w, 0.1, 0.5, ds, dsh, df, da)
    B.pr_head_score(ctx, feat, off, hw, 1, 0.5, rf, hs, hsh, hf)
    B.pr_quantile_score(ctx, feat, off, qw, 0.5, rf, qsum, qs, qsh, qf)


@pytest.mark.parametrize("n,V", [(9, 20000), (200, 9001), (700, 5000)])
def test_inputs_written_just_before_a_call(B, n, V):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x0 = torch.randn(n, V, generator=g, device="cuda").bfloat16()
    ch = torch.randint(0, V, (n,), generator=g, device="cuda", dtype=torch.int32)
    off = torch.tensor([0, n // 3, n // 3, n], dtype=torch.int64, device="cuda")
    feat_np, _ = W.head_features([n], 5)
    f0 = torch.from_numpy(feat_np).cuda()
    hw, qw = torch.from_numpy(W.head_weights(1)).cuda(), torch.from_numpy(W.qmlp_weights()).cuda()
    w = torch.randn(11, generator=g, device="cuda") * 0.1
    f32, u8, i32 = torch.float32, torch.uint8, torch.int32
    spec = [((3,), f32), ((3,), u8), ((3,), i32), ((3, 11), f32), ((n, 8), f32), ((n, 2), i32),
            ((n,), i32), ((3,), f32), ((3,), u8), ((3,), i32), ((3,), f32), ((3,), u8), ((3,), i32),
            ((3, 28), f32), ((n,), f32), ((n,), u8), ((n,), i32), ((n, 11), f32)]
    out = [torch.zeros(s, dtype=d, device="cuda") for s, d in spec]
    ctx = B.pr_ctx_create(0, n, max(n, 3))
    x, feat = x0.clone(), f0.clone()
    args = (B, ctx, x, ch, off, feat, hw, qw, w, out)
    _calls(*args)
    torch.cuda.synchronize()
    ref = [t.clone() for t in out]

    def same():
        return all(np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=a.is_floating_point())
                   for a, b in zip(out, ref))

    for _ in range(10):
        for t in (*out, x, feat):
            t.zero_()
        feat.copy_(f0)
        x.copy_(x0)
        _calls(*args)
        assert same()
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        for t in (*out, x, feat):
            t.zero_()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            x.copy_(x0)
            feat.copy_(f0)
        main.wait_stream(side)
        _calls(*args)
        _calls(*args)
    for _ in range(5):
        graph.replay()
        torch.cuda.synchronize()
        assert same()
    B.pr_ctx_destroy(ctx)


@pytest.mark.parametrize("layers", [1, 2])
def test_head_call_of_rejected_requests_before_a_good_one(B, layers):
    """A head call whose requests are all empty or inconsistent leaves its attention
    grid without work; the calls behind it still wait for its row kernels, which
    write the shared scratch."""
    lengths = [200, 1, 130, 77, 300]
    feat_np, off_np = W.head_features(lengths, 11)
    feat, off = torch.from_numpy(feat_np).cuda(), torch.from_numpy(off_np).cuda()
    n, r = int(off_np[-1]), len(lengths)
    hw = torch.from_numpy(W.head_weights(layers)).cuda()
    empty = torch.full((r + 1,), n, dtype=torch.int64, device="cuda")
    wrong = torch.arange(r + 1, dtype=torch.int64, device="cuda") + n + 1
    ctx = B.pr_ctx_create(0, n, r)
    out = [torch.zeros(r, dtype=d, device="cuda") for d in (torch.float32, torch.uint8, torch.int32)]
    junk = [t.clone() for t in out]
    B.pr_head_score(ctx, feat, off, hw, layers, 0.5, None, *out)
    torch.cuda.synchronize()
    ref = [t.clone() for t in out]

    def calls():
        B.pr_head_score(ctx, feat, off, hw, layers, 0.5, None, *out)
        B.pr_head_score(ctx, -feat, empty, hw, layers, 0.5, None, *junk)
        B.pr_head_score(ctx, feat, wrong, hw, layers, 0.5, None, *junk)
        B.pr_head_score(ctx, feat, off, hw, layers, 0.5, None, *out)

    for _ in range(20):
        calls()
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
    assert (junk[2] == B.PR_FLAG_BAD_OFFSETS).all()
    B.pr_ctx_destroy(ctx)


def _replays_and_calls(run, out, ref, spoil):
    """`run` eagerly and from a captured graph, each time after `spoil`: always `ref`"""
    def same():
        return all(np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=a.is_floating_point())
                   for a, b in zip(out, ref))

    for _ in range(10):
        spoil()
        run()
        assert same()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        spoil()
        run()
    for _ in range(5):
        graph.replay()
        torch.cuda.synchronize()
        assert same()


@pytest.mark.parametrize("n,d,V", [(7, 64, 3000), (130, 128, 9001), (300, 64, 20000)])
def test_lmhead_calls_read_what_was_written_just_before(B, n, d, V):
    """Both LM-head calls back to back on one context (one workspace of states), hidden
    states and weights written by the kernels just before."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    h0 = torch.randn(n, d, generator=g, device="cuda").bfloat16()
    w0 = (torch.randn(V, d, generator=g, device="cuda") * 0.2).bfloat16()
    ch = torch.randint(0, V, (n,), generator=g, device="cuda", dtype=torch.int32)
    slot = torch.arange(n, dtype=torch.int32, device="cuda")
    eos = torch.ones(n, dtype=torch.uint8, device="cuda")
    w = torch.randn(11, generator=g, device="cuda") * 0.1
    off = torch.tensor([0, n // 2, n], dtype=torch.int64, device="cuda")
    f32, u8, i32 = torch.float32, torch.uint8, torch.int32
    spec = [((n, 8), f32), ((n, 2), i32), ((n,), i32), ((n,), f32), ((n,), u8), ((n,), i32),
            ((2, 11), f32), ((2,), f32), ((2,), u8), ((2,), i32)]
    out = [torch.zeros(s, dtype=t, device="cuda") for s, t in spec]
    feat, top2, fl, ds, dsh, df, agg, sc, sh, rf = out
    h, lw = h0.clone(), w0.clone()
    ctx = B.pr_ctx_create(0, n, n)

    def run():
        B.pr_lmhead_features(ctx, h, lw, ch, 20, off, feat, top2, fl)
        B.pr_lmhead_decode_step(ctx, h, lw, slot, ch, eos, w, 0.1, 0.5, ds, dsh, df)
        B.pr_aggregate_score(ctx, feat, off, w, 0.1, 0.5, fl, agg, sc, sh, rf)
        B.pr_lmhead_features(ctx, h, lw, ch, 20, off, feat, top2, fl)

    run()
    torch.cuda.synchronize()
    ref = [t.clone() for t in out]

    def spoil():
        for t in (*out, h, lw):
            t.zero_()
        lw.copy_(w0)
        h.copy_(h0)

    _replays_and_calls(run, out, ref, spoil)
    B.pr_ctx_destroy(ctx)


@pytest.mark.parametrize("n,V,n_req", [(40, 9001, 3), (900, 4000, 40), (3000, 2000, 700)])
def test_scorers_read_the_records_of_the_call_just_before(B, n, V, n_req):
    """The feature call writes the records; pooling, the quantile scorer and the head read
    them at once, and the feature call overwrites them for the next round."""
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    x0 = torch.randn(n, V, generator=g, device="cuda").bfloat16()
    ch = torch.randint(0, V, (n,), generator=g, device="cuda", dtype=torch.int32)
    cut = np.sort(np.random.Generator(np.random.PCG64(n)).integers(0, n, n_req - 1))
    off = torch.from_numpy(np.r_[0, cut, n].astype(np.int64)).cuda()
    hw, qw = torch.from_numpy(W.head_weights(1)).cuda(), torch.from_numpy(W.qmlp_weights()).cuda()
    w = torch.randn(11, generator=g, device="cuda") * 0.1
    f32, u8, i32 = torch.float32, torch.uint8, torch.int32
    out = [torch.zeros(s, dtype=t, device="cuda") for s, t in
           [((n_req, 11), f32), ((n_req, 28), f32)] + 3 * [((n_req,), f32), ((n_req,), u8), ((n_req,), i32)]]
    agg, summ, ps, psh, pf, qs, qsh, qf, hs, hsh, hf = out
    rec = torch.zeros(n, 8, device="cuda")
    top2 = torch.zeros(n, 2, dtype=i32, device="cuda")
    fl = torch.zeros(n, dtype=i32, device="cuda")
    x = x0.clone()
    other = -x0
    ctx = B.pr_ctx_create(0, n, n_req)

    def run():
        for y in (other, x):  # the scores of the first round are overwritten by the second's
            B.pr_token_features(ctx, y, ch, 20, off, rec, top2, fl)
            B.pr_aggregate_score(ctx, rec, off, w, 0.1, 0.5, fl, agg, ps, psh, pf)
            B.pr_token_features(ctx, y, ch, 20, off, rec, top2, fl)
            B.pr_quantile_score(ctx, rec, off, qw, 0.5, fl, summ, qs, qsh, qf)
            B.pr_token_features(ctx, y, ch, 20, off, rec, top2, fl)
            B.pr_head_score(ctx, rec, off, hw, 1, 0.5, fl, hs, hsh, hf)

    run()
    torch.cuda.synchronize()
    ref = [t.clone() for t in out]

    def spoil():
        for t in (*out, rec, x):
            t.zero_()
        x.copy_(x0)

    _replays_and_calls(run, out, ref, spoil)
    B.pr_ctx_destroy(ctx)


def test_selective_metrics_of_scores_written_just_before(B):
    """Scores of the head call ahead of it, and of a kernel; pools of different sizes, which
    share a workspace."""
    ctx = B.pr_ctx_create(0, 16, 4)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    pools = [(torch.rand(n, generator=g, device="cuda"),
              (torch.rand(n, generator=g, device="cuda") < 0.6).to(torch.uint8)) for n in (200000, 900, 70000)]
    ref = [B.pr_selective_metrics(ctx, s, 0.4, labels=y) for s, y in pools]
    for _ in range(5):
        for (s, y), r in zip(pools, ref):
            t = torch.zeros_like(s)
            t.copy_(s)
            assert B.pr_selective_metrics(ctx, t, 0.4, labels=y) == r
    lengths = [50, 3, 700]
    feat_np, off_np = W.head_features(lengths, 3)
    feat, off = torch.from_numpy(feat_np).cuda(), torch.from_numpy(off_np).cuda()
    hw = torch.from_numpy(W.head_weights(1)).cuda()
    score = torch.zeros(3, device="cuda")
    ship, fl = torch.zeros(3, dtype=torch.uint8, device="cuda"), torch.zeros(3, dtype=torch.int32, device="cuda")
    lab = torch.tensor([1, 0, 1], dtype=torch.uint8, device="cuda")
    B.pr_head_score(ctx, feat, off, hw, 1, 0.5, None, score, ship, fl)
    torch.cuda.synchronize()
    r = B.pr_selective_metrics(ctx, score.clone(), 0.5, labels=lab)
    for _ in range(5):
        score.zero_()
        B.pr_head_score(ctx, feat, off, hw, 1, 0.5, None, score, ship, fl)
        assert B.pr_selective_metrics(ctx, score, 0.5, labels=lab) == r
    B.pr_ctx_destroy(ctx)

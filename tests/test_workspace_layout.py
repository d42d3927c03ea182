"""Host-side arithmetic of the workspace layout (runs without a GPU)."""
import pytest


# the fixed array of the allocation-free entry is checked against the end of the forward arrays alone: everything that forming
# log-probabilities touches has to lie before it, also from 32769 rows on, where the mask scan is a pass of its own
@pytest.mark.parametrize("static_scratch", [False, True])
@pytest.mark.parametrize("T", [1, 32768, 32769, 40000, 262145, 2 ** 21])
@pytest.mark.parametrize("d,V", [(64, 300), (64, 32768), (2048, 151936)])
def test_forward_arrays_end_where_the_slab_starts(T, d, V, static_scratch):
    from paper_2512_21450_b200.binding import debug_workspace
    total, forward, row_pos_end = debug_workspace(T, d, V, static_scratch=static_scratch)
    assert 0 < row_pos_end <= forward <= total
    assert forward >= T * (2 * d + 28 + 16 * 16) + (4 * T if T > 32768 else 0)


# the size is promised for any call with at most T rows: it must not fall as T grows, whatever the slab's shape is
@pytest.mark.parametrize("d,V,d_ref", [(64, 300, 0), (256, 4096, 0), (2048, 151936, 0), (3584, 152064, 0), (2048, 400000, 0),
                                       (2048, 600000, 0), (2048, 1100000, 0), (64, 5000000, 0), (2048, 151936, 2048),
                                       (64, 9000, 64), (2048, 300000, 2048), (2048, 600000, 2048), (896, 151936, 0)])
def test_size_does_not_fall_with_more_rows(d, V, d_ref):
    from paper_2512_21450_b200.binding import debug_workspace
    rows = sorted(set(list(range(1, 9000, 61)) + list(range(128, 60000, 1280)) + [32768, 32769, 100000, 2 ** 20]))
    for n_sm in (148, 132):
        last = (0, 0)
        for T in rows:
            now = debug_workspace(T, d, V, d_ref, n_sm=n_sm)[:2]
            assert now[0] >= last[0] and now[1] >= last[1], (T, now, last)
            last = now


# scoring touches the forward arrays alone: a workspace of just those, with a guard behind it, is enough and stays whole
@pytest.mark.gpu
def test_scoring_needs_the_forward_arrays_alone():
    import torch
    from paper_2512_21450_b200 import Context, RLHeadError
    from paper_2512_21450_b200.binding import debug_workspace
    T, V, d = 300, 5000, (256, 512)
    gen = torch.Generator(device="cuda").manual_seed(3)
    H = [torch.randn(T, k, generator=gen, device="cuda").to(torch.bfloat16) for k in d]
    W = [(0.05 * torch.randn(V, k, generator=gen, device="cuda")).to(torch.bfloat16) for k in d]
    tok = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    ctx = Context(0)
    try:
        need = ctx.workspace_bytes(T, d[1], V, scoring=True)
        assert need == debug_workspace(T, d[1], V)[1] < ctx.workspace_bytes(T, d[1], V)
        ws = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
        ctx._ws = ws[:need]
        logp, _ = ctx.rl_token_logprobs_multi(H, W, tok)
        one, _, lse = ctx.rl_token_logprobs(H[1], W[1], tok)
        stats = ctx.rl_shard_logit_stats(H[1], W[1], tok, None, 0, V)
        assert ctx.last_device_status()[0] == 0 and ctx._ws.data_ptr() == ws.data_ptr()
        assert (ws[need:] == 0xA5).all()
        for h, w, lp in zip(H, W, logp):
            z = h.double() @ w.double().T
            want = z.gather(1, tok[:, None].long())[:, 0] - torch.logsumexp(z, 1)
            assert (lp - want).abs().max().item() <= 2e-3
        assert torch.equal(one, logp[1])
        assert (stats[:, 0] + stats[:, 1].log() - lse).abs().max().item() <= 1e-5      # fp32, a few last bits of about 10
        ctx._ws = ws[:need - 1024]
        ctx.lib.rl_set_workspace(ctx.handle, ws.data_ptr(), need - 1024)
        with pytest.raises(RLHeadError) as e:                                           # a little less is refused
            ctx.ensure_workspace = lambda *a, **k: None
            ctx.rl_token_logprobs(H[1], W[1], tok)
        assert e.value.status == 4
    finally:
        ctx.close()

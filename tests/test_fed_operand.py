"""dH passes that form their operand (the gradient with respect to the logits) while they read it: the order on the CPU, the
results on the GPU against the form that makes it in a launch of its own."""
import numpy as np
import pytest


@pytest.mark.parametrize("cta_group,workers", [(2, 74), (1, 148), (2, 66), (2, 5), (1, 3)])
def test_every_chunk_is_formed_once(cta_group, workers):
    from paper_2512_21450_b200.binding import debug_feed_order
    rng = np.random.default_rng(workers)
    sizes = [(1, 64, 256, 1), (5632, 151936, 152064, 4), (360, 151936, 152064, 4), (1732, 151936, 152064, 4), (256, 4096, 4096, 1)]
    for _ in range(60):
        V = int(rng.integers(1, 160000))
        sizes.append((int(rng.integers(1, 12000)), V, -(-V // 256) * 256, int(rng.integers(1, 9))))
    for rows, V, ld, n_tiles in sizes:
        pairs, _ = debug_feed_order(rows, V, ld, n_tiles, cta_group, workers)
        count = np.zeros((-(-rows // 128), -(-ld // 512)), dtype=np.int32)
        np.add.at(count, (pairs[:, 0], pairs[:, 1]), 1)
        assert (count == 1).all(), (rows, V, n_tiles)


# whole waves; helpers; parts without helpers; and sizes where it does not pay
@pytest.mark.parametrize("rows,d_tiles,pays", [(6912, 4, True), (2983, 7, True), (2600, 4, True), (1000, 3, True), (4096, 4, False),
                                               (2000, 4, False), (447, 4, False)])
def test_order_keeps_up_with_the_products(rows, d_tiles, pays):
    from paper_2512_21450_b200.binding import debug_feed_order, debug_schedule
    V, ld, workers = 151936, 152064, 74
    pairs, pay = debug_feed_order(rows, V, ld, d_tiles)
    assert pay == pays
    if not pays:
        return
    units = debug_schedule(rows, 32768, V, d_tiles, n_range=1, n_fastest=1, stream_k=2, cta_group=2, n_workers=workers)
    blocks = sum(int(u[6] - u[5]) for u in units) / workers
    # chunks come at an even pace and are complete after 30 % of the pass: then nobody waits for more than a few percent of it
    at = np.empty((-(-rows // 128), -(-ld // 512)))
    at[pairs[:, 0], pairs[:, 1]] = np.arange(1, len(pairs) + 1) / len(pairs) * 0.3 * blocks
    late, plain = np.zeros(workers), np.zeros(workers)
    for w, mu, _, _, _, kb0, kb1, _ in units:
        tiles = [m for m in (2 * mu, 2 * mu + 1) if m < at.shape[0]]
        plain[w] += kb1 - kb0
        for chunk in range(kb0 // 8, -(-kb1 // 8)):
            late[w] = max(late[w], at[tiles, chunk].max()) + min(8 * chunk + 8, kb1) - max(8 * chunk, kb0)
    assert late.max() <= 1.05 * plain.max() + 16


# rows, d and V as above on the GPU: 512- and 256-column tiles of dH, single CTAs, masked rows, a vocabulary that ends inside a
# chunk (and inside its first half), several slabs, an entropy term; `fed` is what the schedule says of the valid rows
@pytest.mark.gpu
@pytest.mark.parametrize("T,d,V,kw,fed", [
    (2600, 2048, 52000, {}, True), (3000, 1280, 46335, dict(masked=0.3), True), (5000, 896, 27136, dict(ent_coef=0.1), True),
    (1700, 3584, 79105, dict(masked=0.1), True), (1000, 1536, 134656, {}, True), (2700, 1024, 50000, dict(cta_group=1), True),
    (6000, 1024, 44000, dict(rows=3072), True), (4096, 2048, 33000, {}, False),
])
def test_fed_matches_a_launch_of_its_own(T, d, V, kw, fed):
    import torch
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.binding import debug_feed_order
    g = torch.Generator(device="cuda").manual_seed(T + d + V)
    H = torch.randn(T, d, generator=g, device="cuda", dtype=torch.bfloat16)
    W = torch.randn(V, d, generator=g, device="cuda", dtype=torch.bfloat16) * 0.02
    tok = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    tok[:2] = torch.tensor([0, V - 1], device="cuda", dtype=torch.int32)
    old = -torch.rand(T, generator=g, device="cuda") - 9.5
    adv = torch.randn(T, generator=g, device="cuda")
    mask = (torch.rand(T, generator=g, device="cuda") >= kw.get("masked", 0.0)).to(torch.uint8)
    n, cg = int(mask.sum()), kw.get("cta_group", 2)
    slabs = -(-n // kw.get("rows", n))
    slab = n if slabs == 1 else -(-(-(-n // slabs)) // 256) * 256
    wide = -(-d // 512) * 2 * 96 <= -(-d // 256) * 100 and cg == 2
    _, pays = debug_feed_order(slab, V, -(-V // 256) * 256, -(-d // (512 if wide else 256)), cg, 148 // cg)
    assert pays == fed
    out = {}
    for apart in (False, True):
        c = Context(0)
        try:
            c.set_cta_group(cg)
            if "rows" in kw:
                c.set_slab_limits(kw["rows"], -(-V // 256) * 256)
            seen = []
            if apart:   # rows of dW are reported: they come before dH, which then finds its operand made
                c.set_dw_slab_hook(lambda slab_index, lo, hi: seen.append((lo, hi)))
            o = c.rl_policy_loss_fwd_bwd(H, W, tok, old, old, adv, mask, 0.2, 0.2, 0.04, ent_coef=kw.get("ent_coef", 0.0),
                                         dH=torch.full((T, d), float("nan"), device="cuda", dtype=torch.bfloat16),
                                         dW=torch.full((V, d), float("nan"), device="cuda"))
            torch.cuda.synchronize()
            assert c.last_device_status()[0] == 0 and bool(seen) == apart
            out[apart] = o
        finally:
            c.close()
    # the operand is the same to the bit, and so is all that is made of it (rows of dW are added up in another order of slabs)
    assert torch.equal(out[False]["dH"], out[True]["dH"])
    if slab == n:
        assert torch.equal(out[False]["dW"], out[True]["dW"])
    else:
        a, b = out[False]["dW"], out[True]["dW"]
        assert float((a - b).norm() / b.norm()) < 1e-6   # fp32 sums of three addends in another order
    assert torch.isfinite(out[False]["dH"].float()).all() and torch.isfinite(out[False]["dW"]).all()


# dH to the caller's rows beside dW, or by a launch of its own where dW's tiles are few and rows long: the last size on either side of
# the rule in words, in columns and in rows, and several column slabs of which the last is narrow
@pytest.mark.gpu
@pytest.mark.parametrize("T,d,V,kw,beside", [
    (1025, 2048, 300, {}, True), (1025, 2112, 300, {}, False), (1024, 2112, 300, {}, True), (1100, 2112, 2048, {}, False), (1100, 2112, 2100, {}, True),
    (1300, 2112, 700, dict(cta_group=1), False), (1300, 2304, 700, dict(fp32=True), False), (3000, 2304, 1300, dict(limits=(1024, 1024)), False),
])
def test_dH_beside_dW_or_behind(T, d, V, kw, beside):
    import torch
    from paper_2512_21450_b200 import Context
    g = torch.Generator(device="cuda").manual_seed(T + d + V)
    H = torch.randn(T, d, generator=g, device="cuda", dtype=torch.bfloat16)
    W = torch.randn(V, d, generator=g, device="cuda", dtype=torch.bfloat16) * 0.02
    tok = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    old = -torch.rand(T, generator=g, device="cuda") - 5
    adv = torch.randn(T, generator=g, device="cuda")
    mask = (torch.rand(T, generator=g, device="cuda") >= 0.2).to(torch.uint8)
    fp32 = kw.get("fp32", False)
    out, behind = {}, {}
    for hook in (False, True):
        c = Context(0)
        try:
            c.set_cta_group(kw.get("cta_group", 2))
            if "limits" in kw:
                c.set_slab_limits(*kw["limits"])
            if hook:   # dW of the slab that is walked last comes before its dH, which then has a launch of its own
                c.set_dw_slab_hook(lambda slab_index, lo, hi: None)
            c.set_profiling(True)
            o = c.rl_policy_loss_fwd_bwd(H, W, tok, old, old, adv, mask, 0.2, 0.2, 0.04, dH_fp32=fp32,
                                         dH=torch.full((T, d), float("nan"), device="cuda", dtype=torch.float32 if fp32 else torch.bfloat16))
            behind[hook] = c.profile_read()[1][7]
            assert c.last_device_status()[0] == 0
            out[hook] = o
        finally:
            c.close()
    slabs = -(-T // kw["limits"][0]) if "limits" in kw else 1
    assert behind[False] == (0 if beside else slabs) and behind[True] == (1 if beside else slabs)
    assert torch.equal(out[False]["dH"], out[True]["dH"]) and bool(torch.isfinite(out[False]["dH"].float()).all())
    p = torch.softmax(H.float() @ W.float().t(), 1)
    # dH = G W with G's rows proportional to p - onehot(token) (no entropy term): the direction of every row
    ref = (p - torch.nn.functional.one_hot(tok.long(), V)) @ W.float()
    cos = torch.nn.functional.cosine_similarity(out[False]["dH"].float(), ref, dim=1).abs()
    rows = (mask == 1) & (out[False]["dH"].float().norm(dim=1) > 0)
    assert int(rows.sum()) > 0.5 * T and float(cos[rows].min()) > 0.999
    assert float(out[False]["dH"][mask == 0].float().abs().max()) == 0.0

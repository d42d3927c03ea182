"""Schedules for calls with few rows: column ranges chosen by waves, tiles of the ragged last wave cut into parts.  The
distribution itself on the CPU, the passes that use it against the oracle on the GPU."""
import numpy as np
import pytest


@pytest.mark.parametrize("cta_group,workers", [(2, 74), (1, 148), (2, 3), (2, 1)])
def test_cut_tiles_cover_every_block_once(cta_group, workers):
    from paper_2512_21450_b200.binding import debug_schedule
    rng = np.random.default_rng(workers)
    sizes = [(1, 64, 1), (1, 64 * 9, 1), (300, 152064, 4), (2757, 152064, 7), (5000, 152064, 4), (18947, 4160, 5)]
    sizes += [(int(rng.integers(1, 20000)), 64 * int(rng.integers(1, 600)), int(rng.integers(1, 12))) for _ in range(60)]
    for rows, k_len, n_tiles in sizes:
        u = debug_schedule(rows, 32768, k_len, n_tiles, n_range=1, n_fastest=1, stream_k=2, cta_group=cta_group,
                           n_workers=workers)
        m_units, kb = -(-rows // (128 * cta_group)), -(-k_len // 64)
        cover = np.zeros((m_units, n_tiles, kb), dtype=np.int32)
        slots, work = set(), np.zeros(workers, dtype=np.int64)
        for w, mu, c0, c1, ks, kb0, kb1, _ in u:
            assert c1 == c0 + 1 and kb1 > kb0
            cover[mu, c0, kb0:kb1] += 1
            work[w] += kb1 - kb0
            if ks == 0:
                assert kb1 - kb0 == kb                           # a whole tile
            else:
                assert ks not in slots and ks <= 2 * workers     # a slot of its own
                slots.add(ks)
        assert (cover == 1).all()
        # within 8 % of an even split of all blocks plus what one part may be too long by, unless parts would get too short
        even = m_units * n_tiles * kb / workers
        if kb >= 8 * workers:
            assert work.max() <= 1.08 * even + 8, (rows, k_len, n_tiles, work.max(), even)


@pytest.mark.parametrize("cta_group,workers", [(2, 74), (1, 148), (2, 66), (2, 5), (2, 3)])
def test_reader_adds_the_slots_that_were_written(cta_group, workers):
    # 13, 21 and 30 cut tiles on 74 workers: several parts each, and helpers that do the ends of parts
    from paper_2512_21450_b200.binding import debug_schedule, debug_tile_slots
    rng = np.random.default_rng(workers)
    sizes = [(256 * 13, 151936, 1), (256 * 7, 40064, 3), (256 * 10, 40064, 3), (300, 40000, 1), (276, 151936, 4)]
    sizes += [(int(rng.integers(1, 20000)), 64 * int(rng.integers(1, 2400)), int(rng.integers(1, 9))) for _ in range(80)]
    for rows, k_len, n_tiles in sizes:
        u = debug_schedule(rows, rows, k_len, n_tiles, n_range=1, n_fastest=1, stream_k=2, cta_group=cta_group, n_workers=workers)
        wrote = {}
        for w, mu, c0, c1, ks, kb0, kb1, _ in u:
            if ks > 0:
                wrote.setdefault(mu * n_tiles + c0, []).append((kb0, ks - 1))
        read = {}
        for tile, slot in debug_tile_slots(rows, k_len, n_tiles, cta_group, workers):
            read.setdefault(int(tile), []).append(int(slot))
        # the same slots for the same tiles, added in the order of their k-blocks
        assert read == {t: [slot for _, slot in sorted(v)] for t, v in wrote.items()}, (rows, k_len, n_tiles)
    if workers == 74:   # the sizes are what they are meant to be: tiles x parts, and pieces besides
        for rows, k_len, n_tiles, whole in ((256 * 13, 151936, 1, 13 * 5), (256 * 7, 40064, 3, 21 * 3), (256 * 10, 40064, 3, 30 * 2)):
            assert len(debug_tile_slots(rows, k_len, n_tiles)) > whole


# 12, 24 and 7 tiles leave 2 or 4 of 74 workers over (too few for the ends of 70 parts), 8 tiles 2; 32 leave 10, 48 leave 26
@pytest.mark.parametrize("rows,n_tiles,k_len,helped", [(600, 4, 151936, False), (1536, 4, 151936, False), (100, 5, 151936, False),
                                                       (400, 2, 152064, False), (1800, 4, 151936, True), (3072, 4, 151936, True)])
def test_helpers_end_with_the_parts(rows, n_tiles, k_len, helped):
    from paper_2512_21450_b200.binding import debug_schedule
    u = debug_schedule(rows, 32768, k_len, n_tiles, n_range=1, n_fastest=1, stream_k=2, cta_group=2, n_workers=74)
    pieces, work = np.zeros(74, dtype=np.int64), np.zeros(74, dtype=np.int64)
    for w, *_, kb0, kb1, _ in u:
        pieces[w] += 1
        work[w] += kb1 - kb0
    assert (pieces.max() > 1) == helped
    # with 20 k-blocks for the output of each part, nobody is later than a part by more than one more
    cost = work + 20 * pieces
    assert cost.max() <= cost[pieces == 1].max() + 20


@pytest.mark.parametrize("rows,n_tiles,most,expect", [(77, 594, 148, 0.88), (276, 594, 118, 0.9), (2757, 594, 75, 0.9),
                                                      (60, 16, 16, 0.0), (1, 1, 16, 0.0), (4096, 594, 75, 0.9)])
def test_column_ranges_fill_the_machine(rows, n_tiles, most, expect):
    from paper_2512_21450_b200.binding import debug_schedule
    u = debug_schedule(rows, 32768, 2048, n_tiles, n_range=-1000 - most, cta_group=2, n_workers=74)
    m_units = -(-rows // 256)
    cover, work = np.zeros((m_units, n_tiles), dtype=np.int32), np.zeros(74, dtype=np.int64)
    for w, mu, c0, c1, *_ in u:
        cover[mu, c0:c1] += 1
        work[w] += c1 - c0
    assert (cover == 1).all() and len({(r[2], r[3]) for r in u}) <= most
    assert work.mean() >= expect * work.max()          # 594 tiles on 74 workers: 9 each at best, 8.03 on average


# T: one 128-row tile (single CTAs form the logits), one and several pairs; V and d: ranges of a few and of many k-blocks,
# tiles of 256 and of 512 columns; masked rows make the valid ones fewer than T says
@pytest.mark.gpu
@pytest.mark.parametrize("L_max,d,V,kw", [
    (1, 64, 300, {}), (16, 64, 70001, {}), (16, 512, 9000, {}), (40, 320, 5000, {}), (150, 768, 40000, {}),
    (150, 1024, 3000, {}), (400, 512, 90000, {}), (40, 512, 9000, dict(cta_group=1)), (150, 512, 40000, dict(max_ctas=10)),
])
@pytest.mark.parametrize("f32", [False, True])
def test_few_rows_match_oracle(L_max, d, V, kw, f32):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    from tests.test_gpu_parity import _check_against_oracle
    c = Context(0)
    try:
        if "cta_group" in kw:
            c.set_cta_group(kw["cta_group"])
        if "max_ctas" in kw:
            c.set_max_ctas(kw["max_ctas"])
        _check_against_oracle(c, make_workload(1, prompts=1, L_max=L_max, d=d, V=V, seed=4000 + V + L_max), dH_fp32=f32)
    finally:
        c.close()


# tiles cut into two and more parts whose ends helpers do: the reader adds up a part, the pieces of its end, the next part
@pytest.mark.gpu
@pytest.mark.parametrize("L_max,d,V,max_ctas,tiles,parts", [(90, 512, 40000, 10, 2, 2), (400, 1536, 40000, 0, 21, 3),
                                                           (500, 1536, 40000, 0, 30, 2), (200, 512, 60000, 18, 4, 2)])
def test_helped_parts_match_oracle(L_max, d, V, max_ctas, tiles, parts):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.binding import debug_schedule
    from paper_2512_21450_b200.workloads import make_workload
    from tests.test_gpu_parity import _check_against_oracle
    w = make_workload(1, prompts=1, L_max=L_max, d=d, V=V, seed=5000 + V + L_max)
    u = debug_schedule(w.n_valid, w.T, V, -(-d // 512), n_range=1, n_fastest=1, stream_k=2, cta_group=2,
                       n_workers=(max_ctas or 148) // 2)
    cut = [r for r in u if r[4] > 0]
    # the case is what it says: so many tiles in so many parts, and more pieces than that
    assert len({(r[1], r[2]) for r in cut}) == tiles and len(cut) > tiles * parts, (w.n_valid, len(cut))
    assert sum(1 for r in cut if r[4] <= tiles * parts) == tiles * parts
    c = Context(0)
    try:
        c.set_max_ctas(max_ctas)
        _check_against_oracle(c, w, dH_fp32=True)
    finally:
        c.close()


# dW of few rows on eight epilogue warps, stored and added to what was there (whose next tile is then on its way to L2): one and
# several tiles per worker, a ragged last row tile and last column tile, K of one to ten blocks, a grid of few workers
@pytest.mark.gpu
@pytest.mark.parametrize("L_max,d,V,kw", [(2, 256, 80000, {}), (20, 320, 50001, {}), (75, 704, 33000, {}), (80, 1024, 20300, {}),
                                         (40, 512, 9000, dict(max_ctas=6))])
def test_dw_of_few_rows_adds_to_what_was_there(L_max, d, V, kw):
    import torch
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    from tests.test_gpu_parity import _check_against_oracle
    w = make_workload(1, prompts=1, L_max=L_max, d=d, V=V, seed=6000 + V + L_max)
    c = Context(0)
    try:
        c.set_max_ctas(kw.get("max_ctas", 0))
        assert w.T <= 640 and -(-V // 256) * -(-d // 256) >= 2 * (kw.get("max_ctas", 148))
        _check_against_oracle(c, w)
        _, adv = c.rl_grpo_advantages(w.rewards, w.G, seq_offsets=w.seq_offsets, T=w.T)
        args = (w.H, w.W, w.tokens, w.old_logp, w.ref_logp, adv, w.mask, w.eps_low, w.eps_high, w.beta)
        plain = c.rl_policy_loss_fwd_bwd(*args)["dW"]
        before = torch.randn(V, d, device="cuda") * float(plain.abs().max())
        added = c.rl_policy_loss_fwd_bwd(*args, dW=before.clone(), accumulate_dW=True)["dW"]
        torch.cuda.synchronize()
        assert torch.equal(added, before + plain)   # one fp32 addition per entry
    finally:
        c.close()

"""GPU parity of crf_decode_step: the first generated tokens on a recovered, mixed-version cache.

Two requests share a page pool; each cache is built under adapter version 0 and then recovered on
window [1, 3) under version 1, so layers hold caches of different versions. Four generation steps
follow, teacher-forced with the oracle's greedy tokens (the first from the first-step logits of the
recovered cache): at every step the device logits must match the oracle's (KL <= 1e-3), the device's
greedy token must match wherever the oracle's top-2 margin is clear, the K/V the step wrote into each
layer's page slot must match the oracle's, and every other slot of the pool stays bit-identical.
"""
import numpy as np
import pytest
import torch

import synth
from tests.harness import DeviceAdapter, DeviceModel, make_pool, pages_needed, split_page_tables
from oracle import cache as C, decoder as Dec, fidelity
from tests.gpu_util import KL_ABS, REL_KVH, oracle_adapter, oracle_model, oracle_pool, rel_frob, snapshot, to_np

pytestmark = pytest.mark.gpu

STEPS = 4


def test_decode_steps_match_oracle():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    cfg, lc = synth.TINY, synth.LORA_TINY
    N = cfg.n_layers
    ns = [300, 77]
    s, e = 1, 3
    dm = DeviceModel(cfg)
    v0, v1 = DeviceAdapter(cfg, lc, 0), DeviceAdapter(cfg, lc, 1)
    P = sum(pages_needed(n + STEPS) for n in ns) + 4
    pts = split_page_tables([n + STEPS for n in ns], P, seed=6)
    pool = make_pool(cfg, P, fill="random", seed=9)
    ctx = crf.Context(0)
    opool = oracle_pool(pool)
    toks = [synth.token_ids(cfg, n, request=i, device="cuda") for i, n in enumerate(ns)]

    # GPU: stale build under v0, recovery under v1 (checkpoints kept for the window restart)
    H = [[torch.empty(n, cfg.hidden, dtype=torch.bfloat16, device="cuda") for _ in range(N)] for n in ns]
    for i, n in enumerate(ns):
        req = crf.Request(pts[i], 0, N, n_tokens=n, tokens=toks[i], hidden_out=H[i])
        ctx.recompute_window(dm.crf, v0.crf, pool, [req], ctx.workspace(dm.crf, v0.crf, [req]))
        req = crf.Request(pts[i], s, e, n_tokens=n, hidden_in=H[i][s - 1], hidden_out=H[i][s:e])
        ctx.recompute_window(dm.crf, v1.crf, pool, [req], ctx.workspace(dm.crf, v1.crf, [req]))
    ctx.check()

    # oracle: the same two steps on its own caches, then the first-step token of each request
    om, oa0, oa1 = oracle_model(dm), oracle_adapter(v0), oracle_adapter(v1)
    oreqs, first = [], []
    for i, n in enumerate(ns):
        oreq = C.RequestCache(to_np(toks[i]).astype(np.int64), pts[i].cpu().numpy())
        C.prefill(om, oa0, opool, oreq)
        _, h_last = C.recover(om, oa1, opool, oreq, s, e)
        oreqs.append(oreq)
        first.append(int(np.argmax(C.logits(om, h_last))))

    before_k, before_v = snapshot(pool)
    ws = ctx.decode_workspace(dm.crf, v1.crf, ns, pts, torch.tensor(first, dtype=torch.int32, device="cuda"))
    cur = list(first)
    for step in range(STEPS):
        pos = [n + step for n in ns]
        tok_dev = torch.tensor(cur, dtype=torch.int32, device="cuda")
        nxt = torch.empty(len(ns), dtype=torch.int32, device="cuda")
        logits = torch.empty(len(ns), cfg.vocab, dtype=torch.float32, device="cuda")
        ctx.decode_step(dm.crf, v1.crf, pool, pos, pts, tok_dev, nxt, ws, logits=logits)
        ctx.check()
        got_z, got_t = to_np(logits).astype(np.float64), to_np(nxt)
        for i in range(len(ns)):
            x = np.asarray(om.embed[cur[i]], np.float32).reshape(1, -1)
            pt = oreqs[i].page_table
            for l in range(N):
                kh, vh = opool.read(l, pt, pos[i])
                x, k, v = Dec.decode_row(x, pos[i], kh, vh, om.layers[l], oa1.layers[l], om.dims)
                opool.k[l][pt[pos[i] // 16], :, pos[i] % 16, :] = k
                opool.v[l][pt[pos[i] // 16], :, pos[i] % 16, :] = v
                page, off = int(pt[pos[i] // 16]), pos[i] % 16
                assert rel_frob(to_np(pool.k_pages[l][page, :, off, :]), k) <= REL_KVH, (step, i, l, "k")
                assert rel_frob(to_np(pool.v_pages[l][page, :, off, :]), v) <= REL_KVH, (step, i, l, "v")
            z = np.asarray(C.logits(om, x[0]), np.float64).reshape(-1)
            assert fidelity.kl(z[None], got_z[i][None])[0] <= KL_ABS, (step, i)
            top = np.sort(z)
            if top[-1] - top[-2] > 0.05:
                assert int(got_t[i]) == int(np.argmax(z)), (step, i)
            cur[i] = int(np.argmax(z))  # teacher forcing with the oracle's greedy token

    # only the generated slots changed
    written = {(int(pts[i][(n + t) // 16]), (n + t) % 16) for i, n in enumerate(ns) for t in range(STEPS)}
    for l in range(N):
        for a, b in ((pool.k_pages[l], before_k[l]), (pool.v_pages[l], before_v[l])):
            mask = torch.ones(a.shape[0], a.shape[2], dtype=torch.bool, device="cuda")
            for page, off in written:
                mask[page, off] = False
            assert torch.equal(a.permute(0, 2, 1, 3)[mask], b.permute(0, 2, 1, 3)[mask])


def test_decode_step_rejects_bad_arguments():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    from paper_2609_30884_gb300.abi import CrfError
    cfg, lc = synth.TINY, synth.LORA_TINY
    dm = DeviceModel(cfg)
    ad = DeviceAdapter(cfg, lc, 1)
    P = 8
    pool = make_pool(cfg, P)
    ctx = crf.Context(0)
    pt = torch.arange(4, dtype=torch.int32, device="cuda")
    tok = torch.zeros(2, dtype=torch.int32, device="cuda")
    nxt = torch.empty(2, dtype=torch.int32, device="cuda")
    ws = ctx.decode_workspace(dm.crf, ad.crf, [20, 20], [pt, pt], tok)
    bk, bv = [t.clone() for t in pool.k_pages], [t.clone() for t in pool.v_pages]
    bad = torch.tensor([0, 99], dtype=torch.int32, device="cuda")
    logits = torch.full((2, cfg.vocab), 7.0, dtype=torch.float32, device="cuda")
    nxt.fill_(-5)
    # page tables are checked by the step's first kernel: the same page in two rows, or an id past
    # the pool, makes the step write nothing (pages, logits, tokens) and crf_check report EINVAL
    for pos, pts, t in (([20, 20], [pt, pt], tok), ([20], [bad], tok[:1])):
        ctx.decode_step(dm.crf, ad.crf, pool, pos, pts, t, nxt[:len(pos)], ws, logits=logits[:len(pos)])
        with pytest.raises(CrfError) as ei:
            ctx.check()
        assert ei.value.status == crf.abi.EINVAL
        assert all(torch.equal(a, b) for a, b in zip(pool.k_pages, bk))
        assert all(torch.equal(a, b) for a, b in zip(pool.v_pages, bv))
        assert torch.all(logits == 7.0) and torch.all(nxt == -5)
    with pytest.raises(CrfError):   # workspace too small: refused before anything is enqueued
        ctx.decode_step(dm.crf, ad.crf, pool, [20], [pt], tok[:1], nxt[:1], ws[:256])
    # a valid step on the same workspace afterwards
    ctx.decode_step(dm.crf, ad.crf, pool, [20], [pt], tok[:1], nxt[:1], ws, logits=logits[:1])
    ctx.check()
    assert not torch.all(logits[0] == 7.0) and int(nxt[0]) >= 0


@pytest.mark.parametrize("bad", [2 ** 31 - 1, -2 ** 31, 2 ** 27, 2 ** 26, -1, 60])
def test_far_page_ids_of_cached_keys_are_rejected(bad):
    """A cached page's id far outside the pool (also where its row index, id x 2 heads x 16, would leave 32
    bits): decode attention asks for such a page before the page check has ended. The step and a direct
    reuse write nothing and report CRF_EINVAL, and the same workspace then serves the right ids."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    cfg = synth.TINY
    dm, ad = DeviceModel(cfg), DeviceAdapter(cfg, synth.LORA_TINY, 1)
    P, pos = 60, 700
    pool = make_pool(cfg, P, fill="random", seed=7)
    ctx = crf.Context(0)
    good = torch.arange(pages_needed(pos + 1), dtype=torch.int32, device="cuda")
    wrong = good.clone()
    wrong[torch.tensor([3, 30], device="cuda")] = bad
    tok = synth.token_ids(cfg, 1, device="cuda")
    h = synth.hidden_state(cfg, pos + 1, device="cuda")
    nxt = torch.full((1,), -5, dtype=torch.int32, device="cuda")
    z = torch.full((1, cfg.vocab), 7.0, device="cuda")
    fin = torch.full((cfg.hidden,), 7.0, dtype=torch.bfloat16, device="cuda")
    ws = ctx.decode_workspace(dm.crf, ad.crf, [pos], [good], tok)

    def reuse(pt):
        req = crf.Request(pt, 2, 2, n_tokens=pos + 1, hidden_in=h, final_hidden_out=fin)
        ctx.recompute_window(dm.crf, ad.crf, pool, [req], ctx.workspace(dm.crf, ad.crf, [req]))

    before = snapshot(pool)
    for call in (lambda: ctx.decode_step(dm.crf, ad.crf, pool, [pos], [wrong], tok, nxt, ws, logits=z), lambda: reuse(wrong)):
        call()
        with pytest.raises(crf.CrfError) as ei:
            ctx.check()
        assert ei.value.status == crf.abi.EINVAL
    assert torch.all(z == 7.0) and int(nxt) == -5 and torch.all(fin == 7.0)
    assert all(torch.equal(a, b) for a, b in zip(pool.k_pages + pool.v_pages, before[0] + before[1]))
    reuse(good)
    ctx.decode_step(dm.crf, ad.crf, pool, [pos], [good], tok, nxt, ws, logits=z)
    ctx.check()
    assert int(nxt) == int(z.argmax()) and torch.all(torch.isfinite(z)) and not torch.all(fin == 7.0)
    ctx.close()


def test_chunk_boundary_positions_do_not_stall():
    """Rows whose position opens a new 128-key chunk (it holds only the row's own key), each streamed
    by blocks of three chunks: the empty chunk reuses a stage whose copies are long consumed, and no
    wait is left for them (a wait for a passed phase runs into the 2 s limit at every layer). Logits and
    the slots written (each opens a page) against the oracle for some of the rows."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import time
    import paper_2609_30884_gb300 as crf
    cfg, lc = synth.TINY, synth.LORA_TINY
    rows, pos = 32, 640
    dm, ad = DeviceModel(cfg), DeviceAdapter(cfg, lc, 1)
    P = rows * pages_needed(pos + 1) + 3
    pts = split_page_tables([pos + 1] * rows, P, seed=8)
    pool = make_pool(cfg, P, fill="random", seed=4)
    ctx = crf.Context(0)
    tok = synth.token_ids(cfg, rows, device="cuda")
    nxt = torch.empty(rows, dtype=torch.int32, device="cuda")
    logits = torch.empty(rows, cfg.vocab, device="cuda")
    ws = ctx.decode_workspace(dm.crf, ad.crf, [pos] * rows, pts, tok)
    opool = oracle_pool(pool)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ctx.decode_step(dm.crf, ad.crf, pool, [pos] * rows, pts, tok, nxt, ws, logits=logits)
    ctx.check()
    assert time.perf_counter() - t0 < 1.5
    om, oa = oracle_model(dm), oracle_adapter(ad)
    for i in (0, 13, rows - 1):
        page, x = int(pts[i][pos // 16]), C.embed(om, [int(tok[i])])
        for l in range(cfg.n_layers):
            kh, vh = opool.read(l, pts[i].cpu().numpy(), pos)
            x, k, v = Dec.decode_row(x, pos, kh, vh, om.layers[l], oa.layers[l], om.dims)
            assert rel_frob(to_np(pool.k_pages[l][page, :, pos % 16]), k) <= REL_KVH, (i, l, "k")
            assert rel_frob(to_np(pool.v_pages[l][page, :, pos % 16]), v) <= REL_KVH, (i, l, "v")
        assert rel_frob(to_np(logits[i]), C.logits(om, x[0])[0]) <= REL_KVH, i
    ctx.close()


@pytest.mark.parametrize("rows,longest", [(3, 40), (9, 1500), (32, 700), (32, 5000)])
def test_rows_of_a_batch_match_the_row_alone(rows, longest):
    """A generation step of many rows (uneven lengths, some below one chunk, one at its edge, one with an
    empty cache; whole runs of chunks per row and, for the longest, runs that cross rows) against
    each row alone. Two roundings part them: a row alone enters the weight passes as three bf16 terms, in
    a batch as two (2^-17 of each input), and its softmax weights are rounded to bf16 relative to running
    maxima that depend on how its chunks are dealt out, so two runs' weights differ by at most 2 x 2^-9
    of themselves and an attention output by at most 2^-8 of its weighted |v|: 2^-6 of the logits'
    norm over four layers if every rounding went the same way. They do not: so many independent roundings
    leave both runs' errors against 64 bits alike (1e-3 to 2e-3, the batch's at most 1.19 times the row
    alone's in 21 rows), so the batch's may be half as large again, plus the two-term inputs (2^-17 each,
    in two passes of a layer that meet its residual: 2^-16; 5e-6 where the cache is empty)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    cfg, lc = synth.TINY, synth.LORA_TINY
    dm, ad = DeviceModel(cfg), DeviceAdapter(cfg, lc, 1)
    pos = [max(0, (longest * (rows - i)) // rows - 3 * i) for i in range(rows)]
    pos[1], pos[-1] = 128 * (pos[1] // 128), 0
    P = sum(pages_needed(p + 1) for p in pos) + 3
    pts = split_page_tables([p + 1 for p in pos], P, seed=21)
    pool = make_pool(cfg, P, fill="random", seed=22)
    before, opool = snapshot(pool), oracle_pool(pool)
    ctx = crf.Context(0)
    tok = synth.token_ids(cfg, rows, device="cuda")

    def step(idx):
        t = tok[idx].contiguous()
        nxt = torch.empty(len(idx), dtype=torch.int32, device="cuda")
        z = torch.empty(len(idx), cfg.vocab, device="cuda")
        p, tables = [pos[i] for i in idx], [pts[i] for i in idx]
        ctx.decode_step(dm.crf, ad.crf, pool, p, tables, t, nxt, ctx.decode_workspace(dm.crf, ad.crf, p, tables, t), logits=z)
        ctx.check()
        assert torch.equal(nxt.long(), z.argmax(-1))
        return z

    z = step(list(range(rows)))
    got_k, got_v = snapshot(pool)
    for pages, old in zip(pool.k_pages + pool.v_pages, before[0] + before[1]):
        pages.copy_(old)
    om, oa = oracle_model(dm), oracle_adapter(ad)
    for i in range(0, rows, max(1, rows // 5)):
        alone = step([i])[0]
        assert (z[i] - alone).norm() <= 2.0 ** -6 * alone.norm(), (i, pos[i])
        x = C.embed(om, [int(tok[i])], np.float64)
        for l in range(cfg.n_layers):
            kh, vh = opool.read(l, pts[i].cpu().numpy(), pos[i])
            x, _, _ = Dec.decode_row(x, pos[i], kh, vh, om.layers[l], oa.layers[l], om.dims, np.float64)
        want = C.logits(om, x[0], np.float64)[0]
        assert rel_frob(to_np(z[i]), want) <= 1.5 * rel_frob(to_np(alone), want) + 2.0 ** -16, (i, pos[i])
    # every slot but the rows' own is untouched
    own = torch.zeros(P, 16, dtype=torch.bool, device="cuda")
    for p, pt in zip(pos, pts):
        own[int(pt[p // 16]), p % 16] = True
    for new, old in zip(got_k + got_v, before[0] + before[1]):
        m = ~own[:, None, :, None].expand_as(new)
        assert torch.equal(new[m], old[m])
    ctx.close()


@pytest.mark.parametrize("vocab,rows", [(4096, 1), (4097, 2), (9001, 3), (20000, 32)])
def test_greedy_token_over_several_blocks(vocab, rows):
    """The greedy token where a row's logits are shared by several blocks (one at 4096, a second with
    one logit at 4097, several with a ragged last one): equal LM head rows spread over all blocks tie for
    the maximum and the lowest index wins; a NaN logit (a NaN in the LM head's first row) never does. With
    every LM head row zero all logits are zeros of both signs, and token 0 wins."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    cfg, lc = synth.replace(synth.TINY, vocab=vocab), synth.LORA_TINY
    dm, ad = DeviceModel(cfg), DeviceAdapter(cfg, lc, 1)
    pos = [5 + i for i in range(rows)]
    P = sum(pages_needed(p + 1) for p in pos)
    pts = split_page_tables([p + 1 for p in pos], P, seed=5)
    pool = make_pool(cfg, P, fill="random", seed=6)
    ctx = crf.Context(0)
    tok = synth.token_ids(cfg, rows, device="cuda") % vocab

    def step():
        nxt = torch.empty(rows, dtype=torch.int32, device="cuda")
        z = torch.empty(rows, vocab, device="cuda")
        ctx.decode_step(dm.crf, ad.crf, pool, pos, pts, tok, nxt,
                        ctx.decode_workspace(dm.crf, ad.crf, pos, pts, tok), logits=z)
        ctx.check()
        return to_np(nxt), to_np(z)

    period = 97  # every block holds copies of every distinct row
    dm.lm_head.copy_(dm.lm_head[:period].repeat(-(-vocab // period), 1)[:vocab].clone())
    dm.lm_head[0, 0] = float("nan")
    nxt, z = step()
    for r in range(rows):
        assert np.isnan(z[r, 0])
        assert np.sum(z[r] == np.nanmax(z[r])) > 1
        assert nxt[r] == np.nanargmax(z[r])
    dm.lm_head.zero_()
    dm.lm_head[::2].neg_()
    nxt, z = step()
    assert np.all(z == 0) and np.all(nxt == 0)
    ctx.close()


@pytest.mark.parametrize("head_dim,hq,hkv", [(64, 7, 1), (64, 14, 2), (64, 16, 2), (128, 7, 1), (128, 16, 2)])
def test_groups_of_seven_and_eight_heads(head_dim, hq, hkv):
    """The largest groups of query heads a KV head has, at both head dimensions: q of the group and the
    row's own k and v are 576 to 1280 elements of a block, whose 256 threads take them in turns. A
    generation step of a row with an empty cache (its own key and value alone make o), one in a chunk's
    middle and one that opens a chunk, then the first-step row of a window, against the oracle: logits,
    the K/V slots written, the final row."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    cfg = synth.replace(synth.TINY, n_layers=2, n_q_heads=hq, n_kv_heads=hkv, head_dim=head_dim, qkv_bias=True)
    dm, ad = DeviceModel(cfg), DeviceAdapter(cfg, synth.LORA_TINY, 1)
    om, oa = oracle_model(dm), oracle_adapter(ad)
    pos = [0, 77, 256]
    P = sum(pages_needed(p + 1) for p in pos) + 3
    pts = split_page_tables([p + 1 for p in pos], P, seed=17)
    pool = make_pool(cfg, P, fill="random", seed=18)
    opool = oracle_pool(pool)
    ctx = crf.Context(0)
    tok = synth.token_ids(cfg, len(pos), device="cuda")
    nxt = torch.empty(len(pos), dtype=torch.int32, device="cuda")
    logits = torch.empty(len(pos), cfg.vocab, device="cuda")
    ws = ctx.decode_workspace(dm.crf, ad.crf, pos, pts, tok)
    ctx.decode_step(dm.crf, ad.crf, pool, pos, pts, tok, nxt, ws, logits=logits)
    ctx.check()
    for i, p in enumerate(pos):
        x, pt = C.embed(om, [int(tok[i])]), pts[i].cpu().numpy()
        page, off = int(pt[p // 16]), p % 16
        for l in range(cfg.n_layers):
            kh, vh = opool.read(l, pt, p)
            x, k, v = Dec.decode_row(x, p, kh, vh, om.layers[l], oa.layers[l], om.dims)
            assert rel_frob(to_np(pool.k_pages[l][page, :, off]), k) <= REL_KVH, (p, l, "k")
            assert rel_frob(to_np(pool.v_pages[l][page, :, off]), v) <= REL_KVH, (p, l, "v")
        z = C.logits(om, x[0])[0]
        assert rel_frob(to_np(logits[i]), z) <= REL_KVH, p
        assert int(nxt[i]) == int(torch.argmax(logits[i]))

    n = 257
    P = pages_needed(n) + 3
    pt = split_page_tables([n], P, seed=19)[0]
    pool = make_pool(cfg, P, fill="random", seed=20)
    opool = oracle_pool(pool)
    tokens = synth.token_ids(cfg, n, request=1, device="cuda")
    fin = torch.empty(cfg.hidden, dtype=torch.bfloat16, device="cuda")
    req = crf.Request(pt, 0, 1, tokens=tokens, final_hidden_out=fin)
    ctx.recompute_window(dm.crf, ad.crf, pool, [req], ctx.workspace(dm.crf, ad.crf, [req]))
    ctx.check()
    oreq = C.RequestCache(to_np(tokens).astype(np.int64), pt.cpu().numpy())
    _, h_last = C.recover(om, oa, opool, oreq, 0, 1)
    assert rel_frob(to_np(fin), h_last) <= REL_KVH
    ctx.close()


@pytest.mark.parametrize("rows", [1, 2])
@pytest.mark.parametrize("shape,limit", [("tiny", 2.6e-7), ("odd", 2.6e-7), ("1.5b", 3.6e-7)])
def test_one_and_two_rows_keep_fp32_sums(shape, limit, rows):
    """One or two rows go through the weight passes at fp32 accuracy. A generation step of one layer with
    empty caches (o is the row's own value, so no weight or key is rounded to bf16) against the oracle in
    64 bits: relative error of the logits. fp32 sums on CUDA cores gave 1.7e-7 (tiny, at most 2.0e-7) and
    2.6e-7 (1.5B shape, at most 2.9e-7) over 16 to 48 rows; running sums that the tensor core cuts off
    over 60 products of 16, 4.7e-7 to 5.6e-7 on the 1.5B shape. The limits leave a fifth over the former's
    largest. "odd": 5 K blocks, and 17 of which the last holds 8 columns, one weight tile past a whole one."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    base, lc = (synth.QWEN15B, synth.LORA_QWEN) if shape == "1.5b" else (synth.TINY, synth.LORA_TINY)
    cfg = synth.replace(base, n_layers=1, vocab=4096)
    if shape == "odd":
        cfg = synth.replace(cfg, hidden=320, ffn=1032, vocab=3001)
    dm, ad = DeviceModel(cfg), DeviceAdapter(cfg, synth.replace(lc, modules=synth.MODULES), 1)
    om, oa = oracle_model(dm), oracle_adapter(ad)
    pool = make_pool(cfg, rows)
    pts = [torch.tensor([i], dtype=torch.int32, device="cuda") for i in range(rows)]
    ctx = crf.Context(0)
    ws = ctx.decode_workspace(dm.crf, ad.crf, [0] * rows, pts, torch.zeros(rows, dtype=torch.int32, device="cuda"))
    none = np.zeros((0, cfg.n_kv_heads, cfg.head_dim))
    for first in (5, 901, 2777):
        tok = torch.arange(first, first + rows, dtype=torch.int32, device="cuda")
        nxt = torch.empty(rows, dtype=torch.int32, device="cuda")
        z = torch.empty(rows, cfg.vocab, device="cuda")
        ctx.decode_step(dm.crf, ad.crf, pool, [0] * rows, pts, tok, nxt, ws, logits=z)
        ctx.check()
        for i in range(rows):
            x = C.embed(om, [first + i], np.float64)
            x, _, _ = Dec.decode_row(x, 0, none, none, om.layers[0], oa.layers[0], om.dims, np.float64)
            assert rel_frob(to_np(z[i]), C.logits(om, x[0], np.float64)[0]) <= limit, (first, i)
    ctx.close()


@pytest.mark.parametrize("rows", [1, 2, 3])
def test_rows_carry_infinities_and_the_largest_values(rows):
    """An MLP activation that overflows gives the row's outputs an infinity of its weights' signs, and one
    between the largest bf16 and the largest fp32 value stays finite: rows enter the weight passes as
    bf16 terms, of which none may be infinity minus infinity. Gate and up of one value, all other weights
    zero, so the first-step row is 1 + w silu(g) u (rounded to bf16; the terms keep 2^-17)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    cfg = synth.replace(synth.TINY, n_layers=1)
    h, dev = cfg.hidden, "cuda"
    sign = torch.where(torch.arange(h, device=dev) % 3 == 0, -1.0, 1.0)
    pool = make_pool(cfg, rows)
    ctx = crf.Context(0)
    ones = torch.ones(cfg.vocab, h, dtype=torch.bfloat16, device=dev)
    dims = dict(n_layers=1, hidden=h, n_q_heads=cfg.n_q_heads, n_kv_heads=cfg.n_kv_heads, head_dim=cfg.head_dim,
                ffn=cfg.ffn, vocab=cfg.vocab, rms_eps=0.0, rope_theta=1e4, qkv_bias=False)
    ad = crf.Adapter(4, 8.0, (), [None])
    for gate, up, down in ((2.0 ** 66, 2.0 ** 66, 1.0), (1.3125 * 2.0 ** 64, 1.5234375 * 2.0 ** 63, 2.0 ** -100)):
        w = {k: torch.zeros_like(v) for k, v in synth.layer_weights(cfg, 0, 0, dev).items()}
        w["ln1"].fill_(1.0)
        w["ln2"].fill_(1.0)
        w["W_gate"][7, 0], w["W_up"][7, 0] = gate, up
        w["W_down"][:, 7] = (down * sign).bfloat16()
        model = crf.Model(dims, [w], ones)
        fin = torch.empty(rows, h, dtype=torch.bfloat16, device=dev)
        reqs = [crf.Request(torch.tensor([i], dtype=torch.int32, device=dev), 0, 0, final_hidden_out=fin[i],
                            tokens=torch.zeros(1, dtype=torch.int32, device=dev)) for i in range(rows)]
        ctx.recompute_window(model, ad, pool, reqs, ctx.workspace(model, ad, reqs))
        ctx.check()
        with np.errstate(over="ignore"):
            act = np.float32(gate) * np.float32(up)
        assert np.isinf(act) == (down == 1.0)
        want = 1.0 + sign.double() * down * float(act)
        for i in range(rows):
            got = fin[i].double()
            if np.isinf(act):
                assert torch.equal(got, want), i
            else:
                assert torch.all((got - want).abs() <= 2.0 ** -8 * want.abs()), i
    ctx.close()

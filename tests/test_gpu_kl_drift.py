"""GPU parity of crf_kl and crf_drift against the oracle."""
import numpy as np
import pytest
import torch

import synth
from tests.harness import DeviceAdapter, DeviceModel
from oracle import cache as C, drift as odrift, fidelity
from tests.gpu_util import DRIFT_REL, KL_ABS, oracle_adapter, oracle_model, rel_frob, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30884_gb300 as crf
    return crf.Context(0)


@pytest.mark.parametrize("rows,vocab,scale", [(1, 1024, 1.0), (3, 152064, 3.0), (4, 151936, 0.2),
                                              (2, 5, 1.0)])
def test_kl_from_logits(ctx, rows, vocab, scale):
    z_ref = synth.normal((rows, vocab), "zref", 0, scale, device="cuda")
    z_cur = z_ref + synth.normal((rows, vocab), "dz", 0, 0.3 * scale, device="cuda")
    out = torch.empty(rows, dtype=torch.float32, device="cuda")
    ws = ctx.kl_workspace(rows, vocab)
    ctx.kl(None, z_ref, z_cur, out, vocab, ws)
    ctx.check()
    want = fidelity.kl(to_np(z_ref).astype(np.float64), to_np(z_cur).astype(np.float64))
    np.testing.assert_allclose(to_np(out), want, atol=KL_ABS, rtol=0)
    np.testing.assert_allclose(to_np(out), want, rtol=1e-3, atol=1e-5)
    # KL(p || p) = 0
    ctx.kl(None, z_ref, z_ref, out, vocab, ws)
    torch.cuda.synchronize()
    assert np.all(np.abs(to_np(out)) < 1e-5)


def _captured_edges(stream, enqueue):
    """(number of nodes, [(from, to, programmatic)] as node indices in capture order) of what ``enqueue``
    puts on ``stream``: captured into a graph that is never launched."""
    import ctypes
    import paper_2609_30884_gb300 as crf
    rt = crf.abi.load()  # linked against the runtime: its symbols resolve through this handle
    P, N = ctypes.c_void_p, ctypes.c_size_t

    def call(name, *args):
        fn = getattr(rt, name)
        fn.restype = ctypes.c_int
        assert fn(*args) == 0, name

    s, graph, n = P(stream.cuda_stream), P(), N()
    stream.synchronize()
    call("cudaStreamBeginCapture", s, ctypes.c_int(2))  # relaxed
    try:
        with torch.cuda.stream(stream):
            enqueue()
    finally:
        call("cudaStreamEndCapture", s, ctypes.byref(graph))
    call("cudaGraphGetNodes", graph, None, ctypes.byref(n))
    nodes = (P * n.value)()
    call("cudaGraphGetNodes", graph, nodes, ctypes.byref(n))
    at = {v: i for i, v in enumerate(nodes)}
    call("cudaGraphGetEdges", graph, None, None, None, ctypes.byref(n))
    src, dst, data = (P * n.value)(), (P * n.value)(), (ctypes.c_uint8 * (8 * n.value))()
    call("cudaGraphGetEdges", graph, src, dst, data, ctypes.byref(n))
    edges = [(at[a], at[b], data[8 * i + 2] != 0) for i, (a, b) in enumerate(zip(src, dst))]  # byte 2: the edge's type
    call("cudaGraphDestroy", graph)
    return len(nodes), edges


@pytest.mark.parametrize("rows", [1, 40])
def test_kl_with_model_head_waits_for_earlier_work(ctx, rows):
    """The LM head pass reads its first weights before its own wait (one row pair, and two passes of
    it): whatever the caller enqueued before the call, such as a kernel that writes the head, must have
    ended when the call's first kernel starts. Shown on the captured graph, without running anything:
    the edge out of the caller's kernel is a full dependency, and the later ones (the pass behind the
    rows' kernel) are programmatic."""
    dm = DeviceModel(synth.TINY, layers=[])
    cfg = synth.TINY
    h = synth.hidden_state(cfg, rows, "href", std=2.0, device="cuda")
    out = torch.empty(rows, dtype=torch.float32, device="cuda")
    ws = ctx.kl_workspace(rows, cfg.vocab, cfg.hidden)
    stream = torch.cuda.Stream()

    def enqueue():
        dm.lm_head.mul_(2)
        ctx.kl(dm.crf, h, h, out, cfg.vocab, ws, stream=stream)

    n, edges = _captured_edges(stream, enqueue)
    assert n >= 5 and len(edges) == n - 1
    sources = {a for a, _, _ in edges} - {b for _, b, _ in edges}
    assert len(sources) == 1
    first = [p for a, _, p in edges if a in sources]
    assert first == [False]
    assert any(p for _, _, p in edges)


@pytest.mark.parametrize("cfg", [synth.TINY, synth.QWEN15B], ids=["tiny", "1.5b"])
def test_kl_with_model_head(ctx, cfg):
    dm = DeviceModel(cfg, layers=[])
    om = oracle_model(dm)
    rows = 2
    h_ref = synth.hidden_state(cfg, rows, "href", std=2.0, device="cuda")
    h_cur = (h_ref.float() + synth.normal((rows, cfg.hidden), "dh", 0, 0.3, device="cuda")).bfloat16()
    out = torch.empty(rows, dtype=torch.float32, device="cuda")
    logits = torch.empty(2 * rows, cfg.vocab, dtype=torch.float32, device="cuda")
    ws = ctx.kl_workspace(rows, cfg.vocab, cfg.hidden)
    ctx.kl(dm.crf, h_ref, h_cur, out, cfg.vocab, ws, logits_out=logits)
    ctx.check()
    zr = C.logits(om, to_np(h_ref))
    zc = C.logits(om, to_np(h_cur))
    assert rel_frob(to_np(logits[:rows]), zr) < 1e-4
    assert rel_frob(to_np(logits[rows:]), zc) < 1e-4
    np.testing.assert_allclose(to_np(out), fidelity.kl(zr, zc), atol=KL_ABS, rtol=0)
    # Eq. 4 certificate on the device logits
    lg = to_np(logits).astype(np.float64)
    bound = 0.25 * np.sum((lg[rows:] - lg[:rows]) ** 2, axis=1)
    assert np.all(to_np(out) <= bound + 1e-4)


@pytest.mark.parametrize("hidden", [64, 192, 1536, 1600, 3584, 8192])
def test_head_logits_of_one_pair_keep_fp32_accuracy(ctx, hidden):
    """Logits of one row pair, from one K block to two steps a group, against 64-bit products of the same
    fp32 rows x g / rms. A chain of c = ceil(hidden / 2048) * 4 MMAs drops at most one unit (2^-23) of its
    running sum at each; the chains, 64 or one per 64 columns if those are fewer, err
    independently, so that sums to at most c / sqrt(chains) units of the logits' norm, below one up to
    here; the division of the norm, the sum's end and the rms factor round by half a unit each: two
    units in all. (Sums of 32 MMAs measure 3.8 at 3584.)"""
    cfg = synth.replace(synth.TINY, hidden=hidden, vocab=5000)
    dm = DeviceModel(cfg, layers=[])
    h = synth.hidden_state(cfg, 2, "one-pair", std=2.0, device="cuda")
    out = torch.empty(1, dtype=torch.float32, device="cuda")
    z = torch.empty(2, cfg.vocab, dtype=torch.float32, device="cuda")
    ctx.kl(dm.crf, h[:1], h[1:], out, cfg.vocab, ctx.kl_workspace(1, cfg.vocab, hidden), logits_out=z)
    ctx.check()
    x = h.double()
    want = (x * torch.rsqrt(x.square().mean(-1, keepdim=True) + cfg.rms_eps) * dm.final_norm.double()) @ dm.lm_head.double().T
    assert (z.double() - want).norm() <= 2 * 2.0 ** -23 * want.norm()


@pytest.mark.parametrize("cfg,lc", [(synth.TINY, synth.LORA_TINY), (synth.QWEN15B, synth.LORA_QWEN)],
                         ids=["tiny-r8", "1.5b-r16"])
def test_drift_matches_oracle(ctx, cfg, lc):
    n = cfg.n_layers
    cur = DeviceAdapter(cfg, lc, 3)
    anchors = {v: DeviceAdapter(cfg, lc, v) for v in (0, 1, 3)}
    # mixed-version cache: every layer has its own anchor
    which = [(0, 1, 3)[l % 3] for l in range(n)]
    out = torch.empty(n, 7, 2, dtype=torch.float32, device="cuda")
    ws = ctx.drift_workspace(_dims_c(cfg), cur.crf.dims_c)
    ctx.drift(_dims_c(cfg), cur.crf, [anchors[a].crf for a in which], out, ws)
    ctx.check()
    got = to_np(out).astype(np.float64)
    oc = oracle_adapter(cur).layers
    ref = np.zeros((n, 7, 2))
    anc_np = {v: oracle_adapter(a).layers for v, a in anchors.items()}
    for l in range(n):
        for j, m in enumerate(synth.MODULES):
            if m not in lc.modules:
                continue
            A0, B0 = anc_np[which[l]][l].AB[m]
            A1, B1 = oc[l].AB[m]
            ref[l, j, 0] = odrift.factored_sq(A0, B0, A1, B1)
            ref[l, j, 1] = odrift.param_sq(A0, B0, A1, B1)
    nz = ref > 0
    assert np.all(got[~nz] == 0)
    rel = np.abs(got[nz] - ref[nz]) / ref[nz]
    assert rel.max() <= DRIFT_REL, f"max rel drift error {rel.max():.3e}"
    # identical versions give exactly zero
    assert np.all(got[[l for l in range(n) if which[l] == 3]] == 0)


def test_drift_more_items_than_one_launch(ctx):
    """240 (layer, module) items, more than one launch pair takes: the host splits them over two
    Gram + combine launches that reuse one workspace. Every adapted entry matches the factored
    oracle (down's 688-wide input ends in a 176-column step, zero-filled past its columns); the
    unadapted v entries, poisoned with NaN first, read zero."""
    cfg = synth.replace(synth.TINY, n_layers=40)
    lc = synth.replace(synth.LORA_TINY, rank=16, modules=("q", "k", "o", "gate", "up", "down"))
    cur, anchor = DeviceAdapter(cfg, lc, 2), DeviceAdapter(cfg, lc, 0)
    out = torch.full((cfg.n_layers, 7, 2), float("nan"), dtype=torch.float32, device="cuda")
    ws = ctx.drift_workspace(_dims_c(cfg), cur.crf.dims_c)
    ctx.drift(_dims_c(cfg), cur.crf, [anchor.crf] * cfg.n_layers, out, ws)
    ctx.check()
    got = to_np(out).astype(np.float64)
    oc, oa = oracle_adapter(cur).layers, oracle_adapter(anchor).layers
    worst = 0.0
    for l in range(cfg.n_layers):
        for j, m in enumerate(synth.MODULES):
            if m not in lc.modules:
                assert got[l, j, 0] == 0.0 and got[l, j, 1] == 0.0, (l, m)
                continue
            A0, B0 = oa[l].AB[m]
            A1, B1 = oc[l].AB[m]
            for k, ref in enumerate((odrift.factored_sq(A0, B0, A1, B1), odrift.param_sq(A0, B0, A1, B1))):
                worst = max(worst, abs(got[l, j, k] - ref) / ref)
    assert worst <= DRIFT_REL, f"max rel drift error {worst:.3e}"


def _dims_c(cfg):
    from paper_2609_30884_gb300 import abi
    return abi.ModelDims(cfg.n_layers, cfg.hidden, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim,
                         cfg.ffn, cfg.vocab, cfg.rms_eps, cfg.rope_theta, int(cfg.qkv_bias))


@pytest.mark.parametrize("rows,vocab,hidden", [(1, 129, 8), (1, 1000, 200), (2, 127, 64), (5, 700, 1536),
                                               (32, 300, 72), (33, 1024, 256)])
def test_head_logits_at_tile_edges(ctx, rows, vocab, hidden):
    """Logits of the weight pass behind crf_kl at the edges of its tiles: vocabularies beside a multiple
    of 128, hidden sizes below and beside a multiple of 64, one and two rows (three bf16 terms a row),
    more (two terms), and more than one pass of 64 rows. Against fp64; the terms keep 24 and 16 mantissa
    bits and the sums are fp32, so the error of a logit is below 2^-15 of the norm of its products."""
    import paper_2609_30884_gb300 as crf
    g = torch.Generator(device="cuda").manual_seed(rows * 1000 + hidden)
    def draw(*shape, std=1.0):
        return (torch.randn(*shape, device="cuda", generator=g) * std).bfloat16()
    head, norm, ref, cur = draw(vocab, hidden, std=0.05), draw(hidden), draw(rows, hidden), draw(rows, hidden)
    dims = dict(n_layers=1, hidden=hidden, n_q_heads=1, n_kv_heads=1, head_dim=64, ffn=8, vocab=vocab, rms_eps=1e-6,
                rope_theta=1e4, qkv_bias=False)
    model = crf.Model(dims, [None], None, norm, head)
    out, z = torch.empty(rows, device="cuda"), torch.full((2 * rows, vocab), float("nan"), device="cuda")
    ctx.kl(model, ref, cur, out, vocab, ctx.kl_workspace(rows, vocab, hidden), logits_out=z)
    ctx.check()
    x = torch.cat((ref, cur)).double()
    x = x * torch.rsqrt(x.square().mean(-1, keepdim=True) + 1e-6) * norm.double()
    want = x @ head.double().T
    scale = x.square() @ head.double().square().T
    assert ((z.double() - want).abs() <= 2.0 ** -15 * scale.sqrt()).all()
    p, q = (torch.log_softmax(t, -1) for t in want.chunk(2))
    assert ((p.exp() * (p - q)).sum(-1) - out.double()).abs().max() <= 1e-3

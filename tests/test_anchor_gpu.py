"""GPU parity of the layers after the anchor layer (vp_decode_gather).

The anchor layer (layer 0 of a recipe) runs vp_decode_step, whose kept sets
-- checked against the oracle by the decode-step tests -- stay on the
device; a later layer (layer 1, its own caches and query) then attends over
every text token and those kept visual tokens.  The reference is the
oracle's anchor_attention with the same kept sets.
"""

import numpy as np
import pytest
import torch

from oracle import vp_oracle as O
from paper_2605_31457_gb300 import workloads as W

from . import vp_harness as Hn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vp(lib):
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    return lib


def small(**kw):
    base = dict(name="small", layers=2, batch=3, heads=28, kv_heads=4, head_dim=128, dtype=W.BF16,
                vis_len=(300, 577, 64), vis_start=(0, 13, 40), text_len=(517, 70, 129), steps=1,
                planted_frac=0.04, seed=21, beta_range=(0.3, 0.9), beta_sink=1.0,
                budget=W.ADAPTIVE_5PCT)
    base.update(kw)
    return W.Recipe(**base)


def _run(vp, r, budget, layout="bhtd", gran=None, corrupt=None):
    """Anchor at layer 0, gather at layer 1; returns (inputs of layer 1, GPU
    out of layer 1, host kept sets per sequence)."""
    budget = dict(budget)
    if gran is not None:
        budget["granularity"] = gran
    gran = budget.get("granularity", 0)
    inp_a = Hn.make_inputs(r, 0)
    inp_b = Hn.make_inputs(r, 1)
    dev_a = Hn.Device(vp, inp_a, budget, layout=layout)
    dev_b = Hn.Device(vp, inp_b, budget, layout=layout)
    try:
        ga = dev_a.run()
        kept, count = dev_a.kept, dev_a.count
        if corrupt is not None:
            kept = kept.clone()
            kept.view(-1)[0] = corrupt
        vp.vp_decode_gather(dev_b.ctx, dev_b.B, dev_b.q, dev_b.kc, dev_b.vc, dev_b.span, dev_b.tl, kept,
                            dev_a.kept_cap, count, dev_b.out, granularity=gran)
        vp.vp_check_errors(dev_b.ctx)
        torch.cuda.synchronize()
        out = dev_b.out.float().cpu().numpy()
    finally:
        dev_a.close()
        dev_b.close()
    sets = [[ga["kept"][b][g][:int(ga["count"][b][g])] for g in range(ga["kept"].shape[1])]
            for b in range(r.batch)]
    return inp_b, out, sets


def _check(inp, out, sets, seqs=None):
    tol = Hn.TOL[inp.recipe.dtype]
    err = 0.0
    for b in (range(inp.recipe.batch) if seqs is None else seqs):
        want = O.anchor_attention(inp.q[b].double().numpy(), inp.k[b].double().numpy(), inp.v[b].double().numpy(),
                                  int(inp.vis_start[b]), int(inp.vis_len[b]), int(inp.text_len[b]), sets[b])
        np.testing.assert_allclose(out[b], want, rtol=0, atol=tol, err_msg=f"seq {b}")
        err = max(err, float(np.abs(out[b] - want).max()))
    return err


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("gran", [0, 1])
def test_anchor_gather_matches_oracle(vp, D, gran):
    r = small(head_dim=D)
    inp, out, sets = _run(vp, r, r.budget, gran=gran)
    _check(inp, out, sets)


@pytest.mark.parametrize("budget", [dict(mode=O.DENSE, tau=0.1), dict(mode=O.FIXED_RATIO, tau=0.1, ratio_ppm=500_000),
                                    dict(mode=O.FIXED_K, tau=0.1, fixed_k=0)])
def test_anchor_gather_budgets(vp, budget):
    """Every visual token kept (dense attention), half kept, none kept."""
    r = small()
    inp, out, sets = _run(vp, r, budget)
    _check(inp, out, sets)


@pytest.mark.parametrize("page_size,layout", [(16, "bhtd"), (64, "bthd"), (8, "bhtd")])
def test_anchor_gather_paged(vp, page_size, layout):
    r = small(batch=4, vis_len=(300, 577, 64, 1000), vis_start=(0, 13, 40, 0), text_len=(517, 70, 129, 33),
              paged=True, page_size=page_size)
    inp, out, sets = _run(vp, r, r.budget, layout=layout)
    _check(inp, out, sets)


@pytest.mark.parametrize("layout", ["bthd", "padded"])
def test_anchor_gather_layouts(vp, layout):
    r = small()
    inp, out, sets = _run(vp, r, dict(mode=O.FIXED_RATIO, tau=0.1, ratio_ppm=200_000), layout=layout)
    _check(inp, out, sets)


def test_anchor_gather_edge_lengths(vp):
    """Empty visual span, one visual token, only the current text token, a
    span after the whole prompt."""
    r = small(batch=5, vis_len=(0, 1, 33, 700, 16), vis_start=(0, 0, 1, 0, 9), text_len=(5, 1, 1, 1, 9))
    for budget in (r.budget, dict(mode=O.DENSE, tau=0.1), dict(mode=O.FIXED_K, tau=0.1, fixed_k=3)):
        inp, out, sets = _run(vp, r, budget)
        _check(inp, out, sets)


def test_anchor_gather_many_sequences(vp):
    rng = np.random.default_rng(40)
    vis = tuple(int(x) for x in rng.integers(64, 700, 40))
    start = tuple(int(x) for x in rng.integers(0, 40, 40))
    text = tuple(int(s) + int(x) for s, x in zip(start, rng.integers(1, 300, 40)))
    r = small(batch=40, vis_len=vis, vis_start=start, text_len=text)
    inp, out, sets = _run(vp, r, dict(mode=O.FIXED_RATIO, tau=0.1, ratio_ppm=100_000))
    _check(inp, out, sets, seqs=range(0, 40, 3))


def test_anchor_gather_reports_a_bad_kept_index(vp):
    """A kept index outside the visual span is skipped by the kernel and
    reported by vp_check_errors; nothing faults."""
    r = small()
    with pytest.raises(vp.VPError) as ei:
        _run(vp, r, dict(mode=O.FIXED_K, tau=0.1, fixed_k=5), corrupt=1_000_000)
    assert ei.value.status == vp.VP_ERR_DEVICE_PRECOND


def test_anchor_gather_unsupported_configurations(vp):
    """fp32 caches and layouts without a tensor-map description are refused
    before anything is enqueued."""
    for r, layout in ((small(dtype=W.FP32, head_dim=64), "bhtd"), (small(), "tbhd"),
                      (small(paged=True, page_size=4), "bhtd")):
        inp = Hn.make_inputs(r, 1)
        dev = Hn.Device(vp, inp, r.budget, layout=layout)
        try:
            st = vp.vp_decode_gather(dev.ctx, dev.B, dev.q, dev.kc, dev.vc, dev.span, dev.tl, dev.kept,
                                     dev.kept_cap, dev.count, dev.out, check=False)
            assert st == vp.VP_ERR_UNSUPPORTED, st
        finally:
            dev.close()


@pytest.mark.parametrize("dtype", [W.BF16, W.FP32])
def test_calls_in_turn_on_one_context(vp, dtype):
    """Decode steps of different layers, and for bf16 gathers over their kept
    sets between them, back to back on one small context (the score kernels'
    outputs in two sets, used in turn): enqueued, and captured as three calls
    in a graph replayed between enqueued ones, every output equals the call
    run alone, bit for bit."""
    r = small(layers=3, dtype=dtype, vis_len=(900, 577, 64), text_len=(517, 1070, 129))
    devs = [Hn.Device(vp, Hn.make_inputs(r, i, t_cap=1700), r.budget, max_seq=1700) for i in range(3)]
    ctx = devs[0].ctx

    def new(d):
        return [torch.full_like(d.out, float("nan")), torch.full_like(d.kept, -7), torch.full_like(d.count, -7),
                torch.full_like(d.mass, float("nan")), torch.full_like(d.out, float("nan"))]

    def call(d, o):
        vp.vp_decode_step(ctx, d.B, d.q, d.kc, d.vc, d.span, d.tl, d.budget, o[0], o[1], d.kept_cap, o[2], o[3])

    def gather(d, kept, count, o):
        if dtype == W.BF16:
            vp.vp_decode_gather(ctx, d.B, d.q, d.kc, d.vc, d.span, d.tl, kept, d.kept_cap, count, o[4])

    def step(outs):
        for i, d in enumerate(devs):
            call(d, outs[i])
            gather(devs[(i + 1) % 3], outs[i][1], outs[i][2], outs[i])

    try:
        want = []
        for i, d in enumerate(devs):
            o = new(d)
            call(d, o)
            torch.cuda.synchronize()
            gather(devs[(i + 1) % 3], o[1], o[2], o)
            torch.cuda.synchronize()
            want.append([t.clone() for t in o])
        runs = [[new(d) for d in devs] for _ in range(3)]
        for outs in runs:
            step(outs)
        captured = [new(d) for d in devs]
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for i, d in enumerate(devs):
                call(d, captured[i])
        mixed = [[new(d) for d in devs] for _ in range(2)]
        graph.replay()
        step(mixed[0])
        graph.replay()
        graph.replay()
        step(mixed[1])
        vp.vp_check_errors(ctx)
        torch.cuda.synchronize()
        for outs in runs + mixed:
            for i in range(3):
                for a, b in zip(outs[i], want[i]):
                    assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i
        for i in range(3):
            for a, b in zip(captured[i][:4], want[i][:4]):
                assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i
    finally:
        for d in devs:
            d.close()


def test_captured_calls_between_enqueued_ones(vp):
    """Calls captured on another stream, and not launched, between calls that
    are enqueued back to back: the enqueued ones still use the score kernels'
    output sets in turn, and equal the call run alone, bit for bit; so do the
    captured ones when their graph runs."""
    r = small(layers=2, vis_len=(900, 577, 64), text_len=(517, 1070, 129))
    devs = [Hn.Device(vp, Hn.make_inputs(r, i, t_cap=1700), r.budget, max_seq=1700) for i in range(2)]
    ctx = devs[0].ctx

    def new(d):
        return [torch.full_like(d.out, float("nan")), torch.full_like(d.kept, -7), torch.full_like(d.count, -7),
                torch.full_like(d.mass, float("nan"))]

    def call(d, o, stream):
        vp.vp_decode_step(ctx, d.B, d.q, d.kc, d.vc, d.span, d.tl, d.budget, o[0], o[1], d.kept_cap, o[2], o[3],
                          stream=stream)

    try:
        want = []
        for d in devs:
            o = new(d)
            call(d, o, None)
            torch.cuda.synchronize()
            want.append(o)
        run, side = torch.cuda.Stream(), torch.cuda.Stream()
        n = 24
        outs = [new(devs[i % 2]) for i in range(n)]
        captured = [[new(devs[(i + j) % 2]) for j in range(1 + i % 2)] for i in range(n)]
        graphs = [torch.cuda.CUDAGraph() for _ in range(n)]
        torch.cuda.synchronize()
        for i in range(n):
            call(devs[i % 2], outs[i], run)
            with torch.cuda.stream(side):
                graphs[i].capture_begin(capture_error_mode="relaxed")
                for j, o in enumerate(captured[i]):
                    call(devs[(i + j) % 2], o, side)
                graphs[i].capture_end()
        torch.cuda.synchronize()
        for g in graphs:
            g.replay()
        vp.vp_check_errors(ctx)
        torch.cuda.synchronize()
        for i in range(n):
            for j, o in [(i, outs[i])] + [(i + j, o) for j, o in enumerate(captured[i])]:
                for a, b in zip(o, want[j % 2]):
                    assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i
    finally:
        for d in devs:
            d.close()


@pytest.mark.parametrize("H,Hkv,D,batch,max_seq,path", [(7, 1, 64, 1, 140_000, 0), (28, 4, 128, 1, 140_000, 0),
                                                        (7, 1, 128, 8, 65_536, 2)])
def test_small_pages_in_long_contexts(vp, H, Hkv, D, batch, max_seq, path):
    """Contexts for long sequences over 8-token pages: calls whose page ids fit
    only in the splits of the whole GPU's plan are served (decode steps on the
    tensor-core kernel, layers after the anchor)."""
    r = small(heads=H, kv_heads=Hkv, head_dim=D, batch=batch, vis_len=(300,) * batch, vis_start=(13,) * batch,
              text_len=tuple(150 + i for i in range(batch)), paged=True, page_size=8)
    inp = Hn.make_inputs(r, t_cap=512)
    dev = Hn.Device(vp, inp, r.budget, max_seq=max_seq, score_path=path)
    try:
        gpu = dev.run()
        vp.vp_decode_gather(dev.ctx, dev.B, dev.q, dev.kc, dev.vc, dev.span, dev.tl, dev.kept, dev.kept_cap, dev.count,
                            dev.out)  # the anchor's set on the anchor's inputs: the same attention
        vp.vp_check_errors(dev.ctx)
        again = dev.out.float().cpu().numpy()
    finally:
        dev.close()
    for b in range(batch):
        Hn.compare_seq(inp, gpu, b, r.budget)
    np.testing.assert_allclose(again, gpu["out"], rtol=0, atol=2e-2)

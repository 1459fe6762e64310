"""The streaming kernel of the smallest batches against the oracle and, bit for bit, against the general kernel
(the SERIAL schedule): outputs, routing, dispatched rows, h and y, and the plan that is reported."""
import numpy as np
import pytest
import torch

import workloads as wl
import paper_2609_21483_b200 as pk
from oracle import cost_model as cm
from parity import check_routing, run_case, to_dev

pytestmark = pytest.mark.gpu


def _kinds(moe):
    return set((np.concatenate([a for a in moe.read_trace() if len(a)])[:, 2] >> 24).tolist())


def _state(moe, T):
    r = {k: v.clone() for k, v in moe.routing(T).items()}
    r.update({k: v.view(torch.int16).clone() for k, v in moe.intermediates(T).items()})
    return r


@pytest.mark.parametrize("T", [1, 2, 7, 8, 9, 13, 16, 17, 27, 32])
@pytest.mark.parametrize("H,I,E,k,S", [(128, 128, 4, 1, 0),        # fewer units than CTAs
                                       (1152, 384, 256, 16, 0),    # k and E at their limits, tiles of every width
                                       (2048, 1408, 12, 3, 2),     # ring used many times over; shared experts: 8 rows and more
                                       (256, 7168, 3, 2, 0),       # long rows of h
                                       (16384, 128, 5, 2, 1),      # one row of x takes 32 KB
                                       (512, 1024, 1, 1, 0)])      # one expert has every token
def test_smallest_batches_match_oracle_and_general_kernel(T, H, I, E, k, S):
    cfg = wl.MoEConfig(f"stream_{T}_{H}", 1000 + E, T=T, H=H, I=I, E=E, k=k, S=S, zipf_s=0.8 if E > 4 else None)
    inp = wl.make_inputs(cfg)
    dev = to_dev(inp)
    moe, out, _ = run_case(cfg, inp=inp, dev_tensors=dev)
    assert moe.plan()["kind"] == pk.PLAN_PHASED
    got = _state(moe, T)
    for sm in (4, 100, moe.geometry()["n_sm"]):      # shares of a few tiles and of many
        moe.set_sm_count(sm)
        for _ in range(3):
            assert torch.equal(moe.forward(dev[0], dev[1]).view(torch.int16), out.view(torch.int16)), sm
    moe.enable_trace(4096)      # its records tell which kernel the rule picks: beyond it this compares the general one with itself
    assert torch.equal(moe.forward(dev[0], dev[1]).view(torch.int16), out.view(torch.int16))
    assert (12 in _kinds(moe)) == (T <= 16 and T * (2 * max(H, I) + 16) <= 212992 - 16384 * (8 if T > 8 else 5))
    moe.enable_trace(0)
    _, general, _ = run_case(cfg, sched=(pk.SCHED_SERIAL, 0, 1, 0), inp=inp, dev_tensors=dev, moe=moe)
    assert torch.equal(out.view(torch.int16), general.view(torch.int16))
    want = _state(moe, T)
    for name in want:
        assert torch.equal(got[name], want[name]), name
    moe.close()


def test_smallest_batches_report_the_plan_of_the_cost_model():
    """Whichever kernel runs, the plan is the arg-min over the candidates for the tables that are set."""
    H, I, E, k = 256, 256, 130, 4
    cfg = wl.MoEConfig("stream_plan", 1200, T=8, H=H, I=I, E=E, k=k)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, E, k, 0, max_tokens=8)
    N = moe.geometry()["n_sm"]
    rng = np.random.default_rng(3)
    seen = set()
    for trial in range(24):
        T, kinds = int(rng.integers(1, 9)), int(rng.choice([4, 5, 6, 7, 15]))
        idx = np.arange(N + 1, dtype=np.float64)
        bw = (10 ** rng.uniform(3.0, 5.5) * np.minimum(idx, rng.uniform(20, 148))).astype(np.float32)
        tf = (10 ** rng.uniform(6, 8.0) * idx ** rng.uniform(0.2, 1.0)).astype(np.float32)
        bw[0], tf[0] = bw[1], tf[1]
        eff, alpha = np.array([1.0, .9, .8, .7], np.float32), float(rng.uniform(0, 0.95))
        tab = cm.CostTables(N, bw, tf, eff, alpha, c_min=2, c_max=N // 2, c_step=2, steal_workers=N // 2, max_segments=1024, kinds=kinds)
        moe.set_cost_tables(bw, tf, eff, alpha, 2, N // 2, 2)
        moe.set_model_options(kinds, -1)
        moe.forward(x[:T].contiguous(), lg[:T].contiguous())
        moe.check()
        tiles = int((moe.routing(T)["counts"] > 0).sum()) * (I // 128 + (H + 255) // 256)
        want, got = cm.plan(tab, T, T * k, H, I, [tiles] * 4, n_experts=E), moe.plan()
        assert (got["kind"], got["c"], got["K"]) == (want.kind, want.c, want.K), (trial, got, want)
        assert got["t_total_us"] == pytest.approx(float(want.t_total), rel=1e-6)
        seen.add(got["kind"])
    assert pk.PLAN_PHASED in seen and len(seen) > 1
    moe.close()


@pytest.mark.parametrize("T", [1, 8, 16])
def test_smallest_batches_in_place_and_captured_between_larger_ones(T):
    """out = x; a CUDA graph of two layers; calls of 1 to 40 tokens in turn on one handle, so that both kernels hand the
    control words to each other: the same bits every time."""
    cfg = wl.MoEConfig(f"stream_mix_{T}", 1300, T=40, H=1024, I=512, E=64, k=4, S=1, zipf_s=0.5)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, cfg.E, cfg.k, cfg.S, max_tokens=40)
    xs, ls = x[:T].contiguous(), lg[:T].contiguous()
    ref = moe.forward(xs, ls).view(torch.int16).clone()
    xe = moe.intermediates(T)["xe"].view(torch.int16).clone()
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(200):      # every launch is looked at: a read of x behind the first write of out is a matter of timing
        buf = xs.clone()
        moe.forward(buf, ls, buf)
        wrong += (buf.view(torch.int16) != ref).sum() + (moe.intermediates(T)["xe"].view(torch.int16) != xe).sum()
    assert wrong.item() == 0
    second = moe.forward(buf, ls).view(torch.int16).clone()
    s, g, o1, o2 = torch.cuda.Stream(), torch.cuda.CUDAGraph(), torch.empty_like(xs), torch.empty_like(xs)
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            moe.forward(xs, ls, o1)
            moe.forward(o1, ls, o2)
    for _ in range(3):
        o2.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(o1.view(torch.int16), ref) and torch.equal(o2.view(torch.int16), second)
    refs = {}
    for i in range(400):
        n = (7 * i) % 40 + 1
        out = moe.forward(x[:n].contiguous(), lg[:n].contiguous()).view(torch.int16)
        assert torch.equal(out, refs.setdefault(n, out.clone())), n
    moe.check()
    moe.close()


@pytest.mark.parametrize("T", [1, 8, 16])
@pytest.mark.parametrize("which", [0, 1, -1])
def test_a_wait_that_gives_up_ends_the_streaming_launch(T, which):
    """The finished h tiles of one active expert are never counted in: the waits for them run out, nobody works on with what
    is not there (the expert's rows of y and the output stay as they were), the launch ends without a second limit, and
    the next ones, the one that was queued behind it included, are right again on either kernel."""
    cfg = wl.MoEConfig(f"stream_fail_{T}", 1400, T=64, H=2048, I=1408, E=24, k=3, S=1)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, cfg.E, cfg.k, cfg.S, max_tokens=64)
    xs, ls = x[:T].contiguous(), lg[:T].contiguous()
    ref64 = moe.forward(x, lg).view(torch.int16).clone()
    ref = moe.forward(xs, ls).view(torch.int16).clone()
    moe.check()
    counts, offsets = (moe.routing(T)[n].cpu().numpy() for n in ("counts", "offsets"))
    active = np.flatnonzero(counts)
    e = active[which]
    y, out = moe.intermediates(T)["y"].view(torch.int16), torch.full_like(xs, -3.0)
    y.fill_(0x7fc1)
    limit_ms, t0, t1 = 100, torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    moe.set_timeout_ms(limit_ms)
    moe.debug_withhold_flag(which % len(active))
    t0.record()
    moe.forward(xs, ls, out)
    t1.record()
    moe.debug_withhold_flag(-1)
    moe.set_timeout_ms(4000)
    assert moe.status() == pk.ERR_TIMEOUT
    assert 60 <= moe.last_timeout_where() <= 65
    assert limit_ms <= t0.elapsed_time(t1) < 2 * limit_ms
    assert (y[offsets[e]:offsets[e + 1]] == 0x7fc1).all() and (out == -3.0).all()
    for _ in range(3):
        assert torch.equal(moe.forward(xs, ls).view(torch.int16), ref)
        assert torch.equal(moe.forward(x, lg).view(torch.int16), ref64)
    moe.check()
    moe.set_timeout_ms(20)      # ... and right behind a failed launch, its host status not yet read
    moe.debug_withhold_flag(which % len(active))
    moe.forward(xs, ls)
    moe.debug_withhold_flag(-1)
    moe.set_timeout_ms(4000)
    assert torch.equal(moe.forward(xs, ls).view(torch.int16), ref)
    assert torch.equal(moe.forward(x, lg).view(torch.int16), ref64)
    assert moe.status() == pk.ERR_TIMEOUT
    moe.debug_withhold_flag(len(active))      # an index that the batch does not reach
    assert torch.equal(moe.forward(xs, ls).view(torch.int16), ref)
    moe.check()
    moe.close()


def test_wait_log_of_the_streaming_kernel_tells_its_sixteen_warps_apart():
    """Every failed wait is in its own warp's slot: the producer's (60), the products' (61, 62, 65), the releasing warp's (64)
    and the combine's (63, thread 0); a barrier is named by its offset among the kernel's barriers."""
    cfg = wl.MoEConfig("stream_log", 1450, T=8, H=2048, I=1408, E=24, k=3)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, cfg.E, cfg.k, cfg.S, max_tokens=8)
    moe.set_timeout_ms(20)
    moe.debug_withhold_flag(0)
    moe.forward(x, lg)
    assert moe.status() == pk.ERR_TIMEOUT
    log = moe.wait_log()
    assert len({r[:2] for r in log}) == len(log) and all(0 <= r[0] < moe.geometry()["n_sm"] for r in log)
    warps = {60: {0}, 61: set(range(8, 16)), 62: set(range(8, 16)), 63: {0}, 64: {1}, 65: set(range(8, 16))}
    assert all(r[1] in warps[r[2]] for r in log), log
    failed = [r for r in log if r[2] == 62]
    assert {r[0] for r in failed if r[1] == 8} and {r[1] for r in failed} == set(range(8, 16))
    places = {60: (128, 256), 61: (0, 128), 64: (256, 272), 65: (272, 288)}      # empty, full, done, freed
    assert all(places[r[2]][0] <= (r[3] & 1023) < places[r[2]][1] for r in log if r[2] in places), log
    assert any(r[5] == 1 for r in log) and moe.last_timeout_where() in {r[2] for r in log if r[5] == 1}
    moe.close()


@pytest.mark.parametrize("T", [1, 8, 9, 16])
@pytest.mark.parametrize("H,I,E,k,S", [(2048, 1408, 12, 3, 2), (128, 128, 4, 1, 0), (1152, 384, 256, 16, 0)])
def test_timeline_of_the_smallest_batches_is_the_streaming_kernels(T, H, I, E, k, S):
    """With a timeline set the same kernel runs, with the same bits, and its records account for every unit of columns of
    both phases, every dispatched row, and every CTA's routing, set-up, wait and combine."""
    cfg = wl.MoEConfig(f"stream_trace_{T}", 1460, T=T, H=H, I=I, E=E, k=k, S=S)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, E, k, S, max_tokens=T)
    ref = moe.forward(x, lg).view(torch.int16).clone()
    moe.enable_trace(512)
    assert torch.equal(moe.forward(x, lg).view(torch.int16), ref)
    moe.check()
    trace = moe.read_trace()
    ev = np.concatenate(trace).astype(np.int64)
    kind, ident = ev[:, 2] >> 24, ev[:, 2] & 0xFFFFFF
    active, n_sm = int((moe.routing(T)["counts"] > 0).sum()), moe.geometry()["n_sm"]
    tiles = ident[kind == 12]
    assert ((tiles & 0xFFFF) >= 1).all() and ((tiles & 0xFFFF) <= 8).all()
    for phase, units in ((0, I // 8), (1, H // 16)):
        assert (tiles[tiles >> 16 == phase] & 0xFFFF).sum() == active * units
    np.testing.assert_array_equal(np.sort(ident[kind == 4]), np.arange(T * (k + S)))
    assert all((kind == q).sum() == n_sm for q in (1, 2, 7, 8)) and set(kind) <= {1, 2, 4, 7, 8, 12}
    from paper_2609_21483_b200 import timeline
    rep = timeline.analyse(trace, {"T": T, "H": H, "I": I, "k": k, "S": S})
    assert 0 < rep["tensor_active"] <= 1 and rep["mean_ctas_gemm"] <= n_sm and rep["gemm_TFLOPs"] > 0
    moe.close()


@pytest.mark.parametrize("T,H,I,E,k,S,streams", [
    (16, 128, 128, 4, 1, 0, True), (17, 128, 128, 4, 1, 0, False),          # the largest batch
    (8, 7168, 512, 64, 8, 0, True),                                           # x leaves six ring slots, to the byte
    (8, 7296, 512, 64, 8, 0, False), (8, 7296, 512, 40, 4, 0, True),          # five: 1.43 GB of experts within reach, 0.72 GB
    (3, 4096, 14464, 6, 4, 1, True), (4, 4096, 14336, 6, 4, 1, True),         # h of one expert leaves six
    (4, 4096, 14464, 6, 4, 1, False), (4, 4096, 14464, 6, 3, 1, True),        # five: 1.78 GB of experts at least, 1.42 GB
    (8, 128, 8064, 2, 1, 0, True), (8, 128, 8192, 2, 1, 0, False),            # no room for five
    (9, 4480, 128, 8, 2, 0, True), (9, 4608, 128, 8, 2, 0, False),            # nine tokens and more: eight slots
    (10, 3968, 128, 8, 2, 0, True), (10, 4096, 128, 8, 2, 0, False)])
def test_which_batches_stream(T, H, I, E, k, S, streams):
    """The kernel that runs on both sides of every line of the rule, told by the timeline's records, and its bits against the
    SERIAL schedule's."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    gu, dn = (torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0, 0.02, generator=gen) for s in ((E + S, 2 * I, H), (E + S, H, I)))
    x = torch.empty((T, H), dtype=torch.bfloat16, device="cuda").normal_(0, 1, generator=gen)
    lg = torch.empty((T, E), device="cuda").normal_(0, 1, generator=gen)
    moe = pk.WeaveMoE(gu, dn, E, k, S, max_tokens=T)
    moe.enable_trace(4096)
    for same in (False, True):      # all tokens on the same experts
        out = moe.forward(x, lg[:1].expand(T, E).contiguous() if same else lg).view(torch.int16).clone()
        moe.check()
        assert (12 in _kinds(moe), 6 in _kinds(moe)) == (streams, not streams)
        moe.set_schedule(pk.SCHED_SERIAL)
        assert torch.equal(moe.forward(x, lg[:1].expand(T, E).contiguous() if same else lg).view(torch.int16), out)
        moe.set_schedule(pk.SCHED_AUTO)
    moe.check()
    moe.close()


def _edge_logits(kind, T, E, rng):
    if kind == "equal":                       # ties decide everything
        return np.full((T, E), rng.standard_normal(), np.float32)
    if kind == "quantised":                   # a few values: ties in one lane (e, e + 32) and across lanes
        return rng.integers(-1, 2, (T, E)).astype(np.float32)
    if kind == "signed_zeros":                # -0 == +0
        lg = np.where(rng.random((T, E)) < 0.5, np.float32(0.0), np.float32(-0.0))
        lg[:, rng.integers(0, E)] = -1.0
        return lg.astype(np.float32)
    if kind == "extreme":                     # the largest finite values of either sign, denormals, zeros
        return rng.choice(np.array([3.4028235e38, -3.4028235e38, 1e-45, -1e-45, 0.0, 1.0], np.float32), (T, E))
    lg = rng.standard_normal((T, E)).astype(np.float32)
    lg[T // 2, rng.integers(0, E)] = {"nan": np.nan, "+inf": np.inf, "-inf": -np.inf}[kind]
    return lg


@pytest.mark.parametrize("T", [1, 8, 9, 16])
@pytest.mark.parametrize("E,k", [(4, 2), (4, 4), (40, 5), (130, 16), (256, 8)])
def test_routing_of_the_smallest_batches_at_the_edges(T, E, k):
    """Ties within a lane and across lanes, signed zeros, the largest finite logits, non-finite ones: indices, permutation
    and counts of the oracle where the logits are finite, and the general kernel's status and bits always."""
    cfg = wl.MoEConfig(f"stream_edge_{T}_{E}", 1470 + E, T=T, H=128, I=128, E=E, k=k)
    inp = wl.make_inputs(cfg)
    x, lg, gu, dn = to_dev(inp)
    moe = pk.WeaveMoE(gu, dn, E, k, 0, max_tokens=T)
    moe.enable_trace(256)      # (its records tell which kernel ran)
    rng = np.random.default_rng(T * 1000 + E)
    for kind in ("equal", "quantised", "quantised", "signed_zeros", "extreme", "nan", "+inf", "-inf"):
        inp.logits[:] = _edge_logits(kind, T, E, rng)
        lg.copy_(torch.from_numpy(inp.logits))
        got = []
        for sched in (pk.SCHED_AUTO, pk.SCHED_SERIAL):
            moe.set_schedule(sched)
            out = moe.forward(x, lg).view(torch.int16).clone()
            assert moe.status() == (0 if np.isfinite(inp.logits).all() else pk.ERR_NONFINITE_LOGITS)
            assert (12 in _kinds(moe)) == (sched == pk.SCHED_AUTO)
            got.append((out, _state(moe, T)))
            if np.isfinite(inp.logits).all():
                check_routing(moe, inp)
        assert torch.equal(got[0][0], got[1][0]), kind
        for name in got[0][1]:
            assert torch.equal(got[0][1][name], got[1][1][name]), (kind, name)
    moe.close()


def test_a_captured_batch_keeps_its_plan_as_the_header_says():
    """Tables set behind a capture: a replay of the streaming kernel reports the plan that was made with the old ones, a replay
    of the general kernel the new arg-min; a direct call the new one, whatever the size."""
    cfg = wl.MoEConfig("stream_graph_plan", 1480, T=40, H=512, I=256, E=16, k=2)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, cfg.E, cfg.k, max_tokens=40)
    N = moe.geometry()["n_sm"]
    moe.set_model_options(1 << pk.PLAN_PHASED, -1)
    want, graphs, refs = {}, {}, {}
    s = torch.cuda.Stream()
    for T in (8, 40):
        xs, ls = x[:T].contiguous(), lg[:T].contiguous()
        refs[T] = (xs, ls, moe.forward(xs, ls).view(torch.int16).clone())
        want[T] = moe.plan()["t_total_us"]
        out = torch.empty_like(xs)
        s.wait_stream(torch.cuda.current_stream())
        graphs[T] = (torch.cuda.CUDAGraph(), out)
        with torch.cuda.stream(s):
            with torch.cuda.graph(graphs[T][0], stream=s):
                moe.forward(xs, ls, out)
    idx = np.arange(N + 1, dtype=np.float32)
    moe.set_cost_tables(1e3 * np.maximum(idx, 1), 1e6 * np.maximum(idx, 1), np.array([1.0, .9, .8, .7], np.float32), 0.5, 2, N // 2, 2)
    for T, (g, out) in graphs.items():
        g.replay()
        torch.cuda.synchronize()
        replayed = moe.plan()["t_total_us"]
        assert torch.equal(out.view(torch.int16), refs[T][2])
        moe.forward(refs[T][0], refs[T][1])
        direct = moe.plan()["t_total_us"]
        assert direct > 10 * want[T] and moe.plan()["kind"] == pk.PLAN_PHASED
        # (the general kernel reads BW and TFLOPS on the device; alpha is an argument of the launch)
        assert replayed == want[T] if T <= 16 else replayed > 10 * want[T]
    moe.check()
    moe.close()


def test_smallest_batches_through_the_other_entry_points():
    """forward_static, forward_host and forward_host_pipelined with batches on both sides of the largest streamed one, in turn,
    plain and captured: the handle's bits."""
    cfg = wl.MoEConfig("stream_entries", 1500, T=40, H=1024, I=512, E=24, k=3, S=1)
    x, lg, gu, dn = to_dev(wl.make_inputs(cfg))
    moe = pk.WeaveMoE(gu, dn, cfg.E, cfg.k, cfg.S, max_tokens=40)
    cut = {T: (x[:T].contiguous(), lg[:T].contiguous()) for T in (1, 8, 9, 16, 17, 40)}
    refs = {T: moe.forward(*c).view(torch.int16).clone() for T, c in cut.items()}
    for T in (1, 40, 8, 8, 16, 17, 9, 1, 16, 40):
        out = torch.zeros_like(cut[T][0])
        pk.forward_static(*cut[T], gu, dn, cfg.E, cfg.k, cfg.S, out=out)
        assert torch.equal(out.view(torch.int16), refs[T]), T
    s, g, outs = torch.cuda.Stream(), torch.cuda.CUDAGraph(), {T: torch.zeros_like(c[0]) for T, c in cut.items()}
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            for T, c in cut.items():
                pk.forward_static(*c, gu, dn, cfg.E, cfg.k, cfg.S, out=outs[T])
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(outs[T].view(torch.int16), refs[T]) for T in cut)
    host = [(T, *[t.cpu().pin_memory() for t in cut[T]], torch.zeros_like(cut[T][0], device="cpu").pin_memory()) for T in (8, 40, 1, 16, 9, 17)]
    for call in (moe.forward_host, moe.forward_host_pipelined):
        for T, xh, lh, oh in host:
            call(xh, lh, oh)
        moe.host_wait()
        torch.cuda.synchronize()
        for T, xh, lh, oh in host:
            assert torch.equal(oh.view(torch.int16), refs[T].cpu()), (call, T)
            oh.zero_()
    moe.check()
    moe.close()


@pytest.mark.parametrize("T", [8, 16])
def test_an_abort_in_the_middle_of_a_long_stream(T):
    """Four CTAs take milliseconds for the layer.  The one that waits for the withheld h gives up after 1 ms while the others are
    among their down tiles: their releasing and product warps are cut short at whatever they wait for, and all of them
    leave together."""
    cfg = wl.MoEConfig(f"stream_abort_{T}", 1510, T=T, H=2048, I=1408, E=64, k=8)
    inp = wl.make_inputs(cfg)
    x, lg, gu, dn = to_dev(inp)
    moe = pk.WeaveMoE(gu, dn, cfg.E, cfg.k, max_tokens=T)
    ref = moe.forward(x, lg).view(torch.int16).clone()
    moe.check()
    active = int((moe.routing(T)["counts"] > 0).sum())
    moe.set_sm_count(4)
    for which in (0, active // 4, active // 2, active - 1):
        out = torch.full_like(x, -3.0)
        moe.set_timeout_ms(1)
        moe.debug_withhold_flag(which)
        moe.forward(x, lg, out)
        moe.debug_withhold_flag(-1)
        moe.set_timeout_ms(4000)
        assert moe.status() == pk.ERR_TIMEOUT
        assert (out == -3.0).all() and 60 <= moe.last_timeout_where() <= 65
        assert torch.equal(moe.forward(x, lg).view(torch.int16), ref)
        moe.check()
    moe.set_sm_count(moe.geometry()["n_sm"])
    assert torch.equal(moe.forward(x, lg).view(torch.int16), ref)
    moe.check()
    moe.close()

"""The edges of the kernels' variants: row lengths, chunks, tiles and layer groups.

Single layers are teacher-forced against the fp64 oracle (tests/parity.py, its
tolerance); a call of several layers must give the bits of its layers one by one,
since both take the same arithmetic in the same order.
"""
import pytest
import torch

import parity
from paper_2606_29563_gb300 import kvec, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2606_29563_gb300 import build as kbuild
    import oracle
    kbuild.build()
    oracle.build()


def _wl(Hkv, g=1, **kw):
    return synth.small_workload(num_kv_heads=Hkv, num_q_heads=Hkv * g, **kw)


# The selection's variants hold rows of 4096, 8192, 16384 and 32768 positions, with up to
# eight KV heads; a member of 40 tokens keeps all.  Budgets around the gather's 64 rows.
@pytest.mark.parametrize("L,Hkv,budget,over", [
    (4095, 1, 63, {}), (4096, 3, 64, {}), (4097, 8, 65, {}), (8192, 5, 128, {}), (8193, 2, 129, {}),
    (16384, 1, 600, {}), (16385, 2, 64, {}), (32768, 1, 192, {}), (32769, 2, 64, {}), (4097, 9, 100, {}),
    (4096, 8, 200, dict(head_budget=1, ada_floor=0.25)), (8193, 3, 100, dict(head_budget=1, ada_floor=0.5)),
    (16385, 2, 300, dict(head_budget=1, ada_floor=0.0)), (4097, 9, 100, dict(head_budget=1, ada_floor=0.25)),
])
def test_row_lengths_of_the_selection(L, Hkv, budget, over):
    assert not parity.run_parity(_wl(Hkv, seqlens=(L, 40), budget=budget, layers=2, **over))


# Pooling runs over chunks of 2048 candidates: its window and its moments cross their edges.
# (From two candidates on: the entropy of one is 0, where x ln x / x - ln x leaves up to
# two ulps of ln x and a relative error means nothing.)
@pytest.mark.parametrize("Lc", [2, 2047, 2048, 2049, 4096, 4099])
@pytest.mark.parametrize("over", [dict(pool_kernel=15), dict(pool_mode=1), dict(head_criterion=1), dict(all_positions=1)])
def test_pooling_chunks(Lc, over):
    tail = 0 if over.get("all_positions") else 32
    assert not parity.run_parity(_wl(3, 2, seqlens=(max(Lc + tail, 33),), budget=40, layers=1, **over))


# Window tiles: row counts of the MMA's N, two-block heads, the window sizes that only the
# general kernel takes, a second group of heads, and units of one, two and four tiles.
@pytest.mark.parametrize("Hkv,g,over", [
    (2, 1, dict(window=8, obs_window=8, ext_window=8)), (3, 2, dict(window=16, obs_window=8, ext_window=16)),
    (2, 3, dict(window=16, obs_window=16, ext_window=16)), (2, 8, dict(window=32, obs_window=8, ext_window=24)),
    (1, 5, dict(window=48, obs_window=32, ext_window=40)), (2, 2, dict(window=12, obs_window=5, ext_window=9)),
    (9, 2, {}), (1, 4, dict(seqlens=(4200,) * 5)), (1, 4, dict(seqlens=(4200,) * 9)), (1, 4, dict(seqlens=(4200,) * 18)),
])
def test_window_variants(Hkv, g, over):
    kw = dict(seqlens=(129, 700, 300), budget=100, layers=1)
    kw.update(over)
    assert not parity.run_parity(_wl(Hkv, g, **kw))


def test_equal_scores_of_all_heads_go_to_the_lower_head():
    """K = 0 with the adaptive fill: every score of every head is the same, so the slots
    filled jointly go to head 0's lowest positions (more equal keys than are ranked one
    by one)."""
    L, Hkv = 4500, 8
    wl = _wl(Hkv, seqlens=(L,), budget=96, layers=1, num_ext_heads=0, head_budget=1, ada_floor=0.25)
    x = synth.make_layer(wl, 0)
    sel = kvec.KvecSelector(kvec.params_from_workload(wl))
    cu = torch.tensor(wl.cu_seqlens, dtype=torch.int32)
    idx, _, _ = sel.select_layer(cu, cu.cuda(), x["q_obs"].cuda(), torch.zeros_like(x["k"]).cuda(), x["v"].cuda(),
                                 sel.new_state(1), wl.budget)
    torch.cuda.synchronize()
    preserved = int(0.25 * 96)
    fill = 96 - 32 - preserved
    own = fill // 4
    for h in range(Hkv):
        n = preserved + own + (Hkv * (fill - own) if h == 0 else 0)
        got = [p for p in idx[0, h].cpu().tolist() if p >= 0]
        assert got == list(range(n)) + list(range(L - 32, L)), h
    sel.close()


def test_a_refused_layer_is_complete_where_its_call_is():
    """A call whose every sequence is refused (its state counts 255 layers) has done the
    scores and the heads' choice when its stream reaches the next work, as another call
    has: they are read back there without a wait in between."""
    wl = _wl(8, seqlens=(16000, 15000), budget=500, layers=1)
    x = {k: v.cuda() for k, v in synth.make_layer(wl, 0).items()}
    cu = torch.tensor(wl.cu_seqlens, dtype=torch.int32)
    cu_dev = cu.cuda()
    views = []
    for layers_done in (0, 255):
        sel = kvec.KvecSelector(kvec.params_from_workload(wl))
        state = sel.new_state(wl.batch)
        state[:, 0] = layers_done
        before, outs = state.clone(), sel.alloc_outputs(wl.batch, wl.budget)
        torch.cuda.synchronize()
        sel.select_layer(cu, cu_dev, x["q_obs"], x["k"], x["v"], state, wl.budget, outs=outs)
        views.append(sel.debug())
        if layers_done:
            with pytest.raises(kvec.KvecError):
                kvec.kvec_sync_status(sel.handle)
            assert torch.equal(state, before)
        sel.close()
    for name in ("htop", "sigma", "pres_bits"):
        assert torch.equal(views[0][name], views[1][name]), name


# Layers per launch: more layers than score arrays, chunks that cross heads and sequences
# (partials by item and by segment), more sequences than the walkers cache, no chain
# kernel (nine heads, long rows), the caller's log-sum-exp, the adaptive fill.
@pytest.mark.parametrize("layers,Hkv,seqlens,over", [
    (70, 2, (300, 33), {}), (33, 8, (1500,), {}), (9, 5, (700, 130, 2900), {}), (3, 1, (65,) * 70, {}),
    (13, 9, (500, 300), {}), (5, 9, (500, 300), dict(head_budget=1, ada_floor=0.25)), (3, 1, (33000, 200), {}),
    (10, 4, (2100, 900), dict(head_budget=1, ada_floor=0.25)),
])
@pytest.mark.parametrize("with_lse", [False, True])
def test_layers_of_one_call_match_layer_by_layer(layers, Hkv, seqlens, over, with_lse):
    wl = _wl(Hkv, 2, seqlens=seqlens, budget=64, layers=layers, **over)
    xs = [{k: v.cuda() for k, v in x.items()} for x in synth.make_layers(wl, min(layers, 6))]
    xs = [xs[l % len(xs)] for l in range(layers)]
    lse = None
    if with_lse:
        # Any statistics will do: both sides take the same.
        lse = [torch.full((wl.batch, wl.window, wl.num_q_heads), 7.0 + 0.1 * l, device="cuda") for l in range(layers)]
    cu = torch.tensor(wl.cu_seqlens, dtype=torch.int32)
    sel = kvec.KvecSelector(kvec.params_from_workload(wl, max_layers=layers))
    st1, st2 = sel.new_state(wl.batch), sel.new_state(wl.batch)
    one = [sel.select_layer(cu, cu.cuda(), x["q_obs"], x["k"], x["v"], st1, wl.budget, lse=lse and lse[l])
           for l, x in enumerate(xs)]
    many = [sel.alloc_outputs(wl.batch, wl.budget) for _ in xs]
    for _ in range(3):   # eager, captured, replayed
        st2.zero_()
        sel.select_layers(cu, cu.cuda(), [x["q_obs"] for x in xs], [x["k"] for x in xs], [x["v"] for x in xs],
                          st2, wl.budget, many, lses=lse)
        torch.cuda.synchronize()
        for a, b in zip(one, many):
            for p, q in zip(a, b):
                assert torch.equal(p, q)
        assert torch.equal(st1, st2)
    sel.close()


# A handle beside a model that leaves little memory: the allocation is tried again with
# shorter rings (8 layers in flight, partials of 2), down to a launch a layer.
@pytest.mark.parametrize("layers,Hkv,seqlens,over", [
    (33, 8, (1500, 700), {}), (32, 2, (9000,), {}), (12, 9, (500, 300), {}), (11, 4, (2100,), dict(head_budget=1, ada_floor=0.25)),
])
def test_short_rings_of_a_full_device_give_the_same(layers, Hkv, seqlens, over):
    wl = _wl(Hkv, 2, seqlens=seqlens, budget=64, layers=layers, **over)
    xs = [{k: v.cuda() for k, v in x.items()} for x in synth.make_layers(wl, 5)]
    xs = [xs[l % len(xs)] for l in range(layers)]
    cu = torch.tensor(wl.cu_seqlens, dtype=torch.int32)
    cu_dev = cu.cuda()
    # Room for 16384 positions and more sequences, so that the rings make up the workspace.
    params = kvec.params_from_workload(wl, max_layers=layers, max_seqlen=16384, max_batch=8)
    got, used = [], []
    for fault in (0, 3):
        free = torch.cuda.mem_get_info()[0]
        try:
            kvec.kvec_set_test_fault(fault)
            sel = kvec.KvecSelector(params)
        finally:
            kvec.kvec_set_test_fault(0)
        used.append(free - torch.cuda.mem_get_info()[0])
        outs = [sel.alloc_outputs(wl.batch, wl.budget) for _ in xs]
        for _ in range(3):   # eager, captured, replayed
            state = sel.new_state(wl.batch)
            sel.select_layers(cu, cu_dev, [x["q_obs"] for x in xs], [x["k"] for x in xs], [x["v"] for x in xs],
                              state, wl.budget, outs)
            torch.cuda.synchronize()
            got.append([t.clone() for o in outs for t in o] + [state.clone(), sel.debug()["Pprime"][:wl.batch]])
        sel.close()
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0][:-1], other[:-1]))
    for s, L in enumerate(wl.seqlens):
        assert all(torch.equal(got[0][-1][s, :, :L - wl.window], g[-1][s, :, :L - wl.window]) for g in got[1:])
    rows = 8 * 16416 * Hkv * 4
    S = min(layers, 32)
    assert used[0] - used[1] > (S - 8) * 4 * rows   # four score rows a slot less


# Kernels are programmatic dependents of what precedes them on the stream; in a caller's
# captured graph that may be a copy, a fill or another stream's kernel, whose results
# they must still see.
@pytest.mark.parametrize("before", ["copy", "fill", "other stream"])
@pytest.mark.parametrize("call", ["decode", "layer"])
def test_captured_calls_see_the_work_before_them(before, call):
    gen = torch.Generator().manual_seed(3)
    rand = lambda *shape: torch.randn(shape, generator=gen).to(torch.bfloat16).cuda()
    L, Hkv, Hq, batch, cap = 8000, 8, 16, 16, 1024
    sel = kvec.KvecSelector(kvec.make_params(Hq, Hkv, max_batch=batch, max_seqlen=8192, max_layers=2))
    if call == "decode":
        q, shape = rand(batch, Hq, 128), (batch, Hkv, cap, 128)
        lens = torch.full((batch,), cap, dtype=torch.int32, device="cuda")
        out = [torch.empty((batch, Hq, 128), device="cuda")]
        run = lambda k, v: sel.decode_attention(q, k, v, lens, out=out[0])
    else:
        q, shape = rand(1, 32, Hq, 128), (L, Hkv, 128)
        cu = torch.tensor([0, L], dtype=torch.int32).pin_memory()
        cu_dev, state, out = cu.cuda(), sel.new_state(1), sel.alloc_outputs(1, 256)

        def run(k, v):
            kvec.kvec_reset(sel.handle, state.data_ptr(), 1, torch.cuda.current_stream().cuda_stream)
            sel.select_layer(cu, cu_dev, q, k, v, state, 256, outs=out)
    k, v, ks, vs = (rand(*shape) for _ in range(4))

    def work():
        if before == "copy":
            k.copy_(ks)
            v.copy_(vs)
        elif before == "fill":
            v.copy_(vs)
            k.zero_()
        else:
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                torch.add(ks, 1.0, out=k)
                torch.add(vs, 1.0, out=v)
            torch.cuda.current_stream().wait_stream(side)
        run(k, v)

    side = torch.cuda.Stream()
    main = torch.cuda.Stream()
    with torch.cuda.stream(main):
        work()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=main):
            work()
        for _ in range(3):
            ks.copy_(rand(*shape))
            vs.copy_(rand(*shape))
            work()
            torch.cuda.synchronize()
            expect = [o.clone() for o in out]
            k.fill_(0.25)
            v.fill_(0.5)
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(expect, out))
    sel.close()

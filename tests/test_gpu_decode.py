"""Decode-time eviction with frozen budgets through the C-ABI against the oracle, in lockstep:
before every cake_decode_step the device's state of the layer (positions, scores, cache rows)
is read back, the oracle takes the same step from that state, and the two results are compared:
positions bit for bit, scores within 1e-3 relative, cache rows bit for bit.  Where the oracle's
two lowest scores lie within 1e-3 of each other the device may evict either (fp32 against
float64)."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import cake_oracle as O
from paper_2503_12491_b200 import binding, synth, harness
from paper_2503_12491_b200.binding import CAKE_POOL_AVG, CAKE_POOL_MAX, CakeError, CAKE_ERR_STATE

pytestmark = pytest.mark.gpu

RTOL = 1e-3
UPDATES = {0: "add", 1: "max", 2: "replace"}


def to_np(t):
    return t.detach().float().cpu().numpy().astype(np.float64)


def read_heads(cake, w, r, l, length, k_cache, v_cache, off):
    """The device's decode state of block (r, l) as oracle DecodeHead objects."""
    pos, sc, sl = (x.cpu().numpy() for x in cake.decode_get_state(r, l, length))
    base = int(off[r * w.n_layers + l])
    cap = length + 1
    heads = []
    for g in range(w.n_kv_heads):
        rows = base + g * cap + torch.from_numpy(sl[g].astype(np.int64)).cuda()
        heads.append(O.DecodeHead(pos[g].astype(np.int64), sc[g][: length - w.window].astype(np.float64),
                                  to_np(k_cache[rows]), to_np(v_cache[rows])))
    return heads


def run_decode(w, steps, update_mode=0, pool_mode=CAKE_POOL_MAX):
    L, R, cu = w.n_layers, len(w.seq_lens), w.cu_seqlens
    qs, ks, vs = harness.device_inputs(w)
    cake = harness.cake_for(w, pool_mode=pool_mode)
    k_out, v_out, poff, ppos = cake.run(qs, ks, vs, cu)
    budgets = cake.get_budgets().cpu().numpy()
    packed = harness.split_blocks(w, ppos, poff)
    k_cache, v_cache, off = cake.decode_begin(ks, vs, update_mode)
    assert cake.status() == 0
    off_h = off.cpu().numpy()
    # ---- the initial state: the compacted positions, the survivors' prefill indicators, the rows
    for r, N in enumerate(w.seq_lens):
        for l in range(L):
            length = int(budgets[r, l])
            heads = read_heads(cake, w, r, l, length, k_cache, v_cache, off_h)
            ref = O.score_layer(to_np(qs[l][r]), to_np(ks[l][:, cu[r]:cu[r + 1]]), gamma=w.gamma,
                                pool_kernel=w.pool_kernel, tau1=w.tau1, tau2=w.tau2,
                                pool_mode="max" if pool_mode == CAKE_POOL_MAX else "avg")
            for g in range(w.n_kv_heads):
                want_pos = packed[r][l][g].cpu().numpy()
                assert np.array_equal(heads[g].positions, want_pos)
                want = ref["indicator"][g][want_pos[: length - w.window]]
                assert np.allclose(heads[g].scores, want, rtol=RTOL, atol=1e-30)
                src = to_np(ks[l][g, cu[r] + torch.from_numpy(want_pos).long().cuda()])
                assert np.array_equal(heads[g].k, src)
    # ---- decode steps
    gen = torch.Generator().manual_seed(w.seed + 17)
    near_ties = 0
    for t in range(steps):
        for l in range(L):
            q_new = (torch.randn(R, w.n_q_heads, w.head_dim, generator=gen) * 1.5).to(w.torch_dtype).cuda()
            k_new = torch.randn(R, w.n_kv_heads, w.head_dim, generator=gen).to(w.torch_dtype).cuda()
            v_new = torch.randn(R, w.n_kv_heads, w.head_dim, generator=gen).to(w.torch_dtype).cuda()
            before = [read_heads(cake, w, r, l, int(budgets[r, l]), k_cache, v_cache, off_h) for r in range(R)]
            cake.decode_step(l, q_new, k_new, v_new, k_cache, v_cache)
            for r, N in enumerate(w.seq_lens):
                length = int(budgets[r, l])
                after = read_heads(cake, w, r, l, length, k_cache, v_cache, off_h)
                for g in range(w.n_kv_heads):
                    G = w.group
                    want, ev = O.decode_step_head(
                        before[r][g], to_np(q_new[r, g * G:(g + 1) * G]), to_np(k_new[r, g]), to_np(v_new[r, g]),
                        N + t, window=w.window, budget=length - w.window, pool_kernel=w.pool_kernel,
                        pool_mode="max" if pool_mode == CAKE_POOL_MAX else "avg", update=UPDATES[update_mode])
                    got = after[g]
                    assert len(got.positions) == length and np.all(np.diff(got.positions) > 0)
                    assert got.positions[-1] == N + t
                    if not np.array_equal(got.positions, want.positions):
                        # the device evicted another entry: only allowed at a near tie of the two
                        # lowest scores (recomputed by the oracle with nothing evicted)
                        full, _ = O.decode_step_head(
                            before[r][g], to_np(q_new[r, g * G:(g + 1) * G]), to_np(k_new[r, g]),
                            to_np(v_new[r, g]), N + t, window=w.window, budget=length, pool_kernel=w.pool_kernel,
                            pool_mode="max" if pool_mode == CAKE_POOL_MAX else "avg", update=UPDATES[update_mode])
                        gone_dev = np.setdiff1d(full.positions, got.positions)
                        assert len(gone_dev) == 1 and len(ev) == 1
                        s_dev = full.scores[np.searchsorted(full.positions, gone_dev[0])]
                        s_orc = full.scores[np.searchsorted(full.positions, ev[0])]
                        assert abs(s_dev - s_orc) <= RTOL * abs(s_orc), (t, l, r, g, s_dev, s_orc)
                        near_ties += 1
                        continue
                    assert np.allclose(got.scores, want.scores, rtol=RTOL, atol=1e-12), (t, l, r, g)
                    assert np.array_equal(got.k, want.k) and np.array_equal(got.v, want.v)
    assert cake.status() == 0
    cake.destroy()
    return near_ties


def test_decode_sixty_four_steps_bf16_gqa():
    w = synth.scaled(synth.workload(3), n_layers=2, n_q_heads=8, n_kv_heads=2, seq_lens=(900, 333),
                     total_budget=2 * 120)
    ties = run_decode(w, steps=64)
    assert ties <= 4


def test_decode_fp32_mha_with_average_pooling():
    w = synth.scaled(synth.workload(1), n_layers=2, seq_lens=(300, 150), total_budget=2 * 60)
    run_decode(w, steps=40, pool_mode=CAKE_POOL_AVG)


@pytest.mark.parametrize("mode", [1, 2])
def test_decode_other_update_readings(mode):
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=4, n_kv_heads=1, seq_lens=(500,),
                     total_budget=100)
    run_decode(w, steps=24, update_mode=mode)


@pytest.mark.parametrize("cluster", ["1", "0"])
def test_decode_large_heads(monkeypatch, cluster):
    """Heads of more than 256 slots are spread over a thread-block cluster; with that form switched
    off a head beyond the 5688 slots that G = 8 leaves in shared memory works in the context's
    global work area.  Both must match the oracle like the one-CTA form does."""
    monkeypatch.setenv("CAKE_DECODE_CLUSTER", cluster)
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=8, n_kv_heads=1, seq_lens=(7000, 400),
                     total_budget=6500, window=16)
    run_decode(w, steps=3)


def test_decode_cluster_form_over_many_steps():
    w = synth.scaled(synth.workload(3), n_layers=2, n_q_heads=8, n_kv_heads=2, seq_lens=(2500, 700),
                     total_budget=2 * 900)
    ties = run_decode(w, steps=24)
    assert ties <= 4


def test_decode_requires_a_finished_prefill():
    w = synth.scaled(synth.workload(1), n_layers=2, seq_lens=(100,), total_budget=2 * 30)
    qs, ks, vs = harness.device_inputs(w)
    cake = harness.cake_for(w)
    cake.begin(w.cu_seqlens)
    cake.score_layer(0, qs[0], ks[0]); cake.allocate(0); cake.evict(0)
    with pytest.raises(CakeError) as e:
        cake.decode_begin(ks, vs)
    assert e.value.code == CAKE_ERR_STATE
    cake.destroy()


@pytest.mark.parametrize("layers,budget,heads", [(1, 130, (4, 4)), (2, 255, (8, 2)), (2, 256, (8, 1)), (2, 513, (8, 2)),
                                                 (2, 2055, (4, 2)), (3, 4097, (2, 1))])
def test_decode_heads_at_the_edges_of_a_cta_share(layers, budget, heads):
    """Heads just below and above the entries one CTA takes, and above the clusters of 8 and 16; with
    two or more layers a step starts while the other layer's step still runs."""
    w = synth.scaled(synth.workload(3), n_layers=layers, n_q_heads=heads[0], n_kv_heads=heads[1],
                     window=16, seq_lens=(budget * 2 + 77,), total_budget=layers * budget)
    ties = run_decode(w, steps=4)
    assert ties <= 1


def test_decode_tensors_off_a_32_byte_boundary_give_the_same_state():
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=8, n_kv_heads=2, seq_lens=(900,), total_budget=300)
    qs, ks, vs = harness.device_inputs(w)
    gen = torch.Generator().manual_seed(5)
    vals = [torch.randn(n * w.head_dim, generator=gen).to(w.torch_dtype).cuda() for n in (8, 2, 2)]
    states = []
    for off in (0, 8):                               # 8 bf16 elements: 16 bytes
        cake = harness.cake_for(w)
        cake.run(qs, ks, vs, w.cu_seqlens)
        k_cache, v_cache, _ = cake.decode_begin(ks, vs)
        q, k, v = (torch.zeros(x.numel() + 8, dtype=x.dtype, device="cuda")[off:off + x.numel()].copy_(x) for x in vals)
        cake.decode_step(0, q, k, v, k_cache, v_cache)
        assert cake.status() == 0
        states.append([x.clone() for x in cake.decode_get_state(0, 0, 300)] + [k_cache.clone(), v_cache.clone()])
        cake.destroy()
    assert torch.equal(states[0][0], states[1][0]) and torch.equal(states[0][2], states[1][2])
    assert torch.allclose(states[0][1], states[1][1], rtol=1e-4, atol=1e-9)
    assert torch.equal(states[0][3], states[1][3]) and torch.equal(states[0][4], states[1][4])


def decode_pair(w, tokens):
    """Two contexts with the same finished prefill and decode cache, and the new rows of every step."""
    qs, ks, vs = harness.device_inputs(w)
    gen = torch.Generator().manual_seed(w.seed + 29)
    shapes = [(w.n_q_heads, 1.5), (w.n_kv_heads, 1.0), (w.n_kv_heads, 1.0)]
    new = [[[(torch.randn(len(w.seq_lens), h, w.head_dim, generator=gen) * s).to(w.torch_dtype).cuda() for h, s in shapes]
            for _ in range(w.n_layers)] for _ in range(tokens)]
    out = []
    for _ in range(2):
        cake = harness.cake_for(w)
        cake.run(qs, ks, vs, w.cu_seqlens)
        out.append((cake, *cake.decode_begin(ks, vs)[:2]))
    torch.cuda.synchronize()
    return out, new


def assert_same_decode_state(w, one, two):
    torch.cuda.synchronize()
    budgets = one[0].get_budgets().cpu().numpy()
    for r in range(len(w.seq_lens)):
        for l in range(w.n_layers):
            a, b = (c[0].decode_get_state(r, l, int(budgets[r, l])) for c in (one, two))
            assert all(torch.equal(x, y) for x, y in zip(a, b)), (r, l)
    assert torch.equal(one[1], two[1]) and torch.equal(one[2], two[2])
    assert one[0].status() == 0 and two[0].status() == 0
    one[0].destroy()
    two[0].destroy()


@pytest.mark.parametrize("layers,budget,streams", [(2, 900, (0, 1)), (3, 300, (0, 1, 0)), (4, 1200, (0, 0, 1, 1))])
def test_decode_layers_on_streams_of_their_own(layers, budget, streams):
    """Every layer is stepped on a fixed stream, the layers of a token interleaved over two of them: the
    same states as with all steps on one stream."""
    w = synth.scaled(synth.workload(3), n_layers=layers, n_q_heads=8, n_kv_heads=2, seq_lens=(budget * 2 + 77,),
                     total_budget=layers * budget)
    (one, two), new = decode_pair(w, tokens=12)
    side = [torch.cuda.Stream(), torch.cuda.Stream()]
    for token in new:
        for l, x in enumerate(token):
            one[0].decode_step(l, *x, *one[1:])
    for token in new:
        for l, x in enumerate(token):
            with torch.cuda.stream(side[streams[l]]):
                two[0].decode_step(l, *x, *two[1:])
    assert_same_decode_state(w, one, two)


def capture(rt, streams, body):
    """The graph of what `body` enqueues, captured on streams[0] with the others forked from it and joined."""
    def ok(res):
        assert int(res[0]) == 0, res[0]
        return res[1:]
    main = streams[0]
    ok(rt.cudaStreamBeginCapture(main.cuda_stream, rt.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal))
    body()
    for s in streams[1:]:
        main.wait_stream(s)
    graph, = ok(rt.cudaStreamEndCapture(main.cuda_stream))
    lib, count = ctypes.CDLL("libcudart.so.12"), ctypes.c_size_t(0)
    handle = ctypes.c_void_p(int(graph))
    assert lib.cudaGraphGetEdges_v2(handle, None, None, None, ctypes.byref(count)) == 0
    nodes, data = [(ctypes.c_void_p * count.value)() for _ in range(2)], (ctypes.c_uint8 * (8 * count.value))()
    assert lib.cudaGraphGetEdges_v2(handle, *nodes, data, ctypes.byref(count)) == 0
    return graph, [data[8 * i + 2] for i in range(count.value)], ok          # (from_port, to_port, type, ...)


def test_captured_decode_steps_start_early_only_behind_another_layers_step():
    """In a capture the early start shows as the type of the edge between two launches (1: the second may
    start before the first has finished).  Steps of two layers in turn on one stream have such edges, and the
    replayed graph gives the states of plain steps; a layer's step right behind its own previous one, with
    the other layer on another stream, has none."""
    rt = pytest.importorskip("cuda.bindings.runtime")
    w = synth.scaled(synth.workload(3), n_layers=2, n_q_heads=8, n_kv_heads=2, seq_lens=(1900,), total_budget=2 * 900)
    (one, two), new = decode_pair(w, tokens=4)
    for token in new:
        for l, x in enumerate(token):
            one[0].decode_step(l, *x, *one[1:])
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):                        # outside a capture first: kernel attributes are set then
        for l in range(2):
            two[0].decode_step(l, *new[0][l], *two[1:])
        torch.cuda.synchronize()

    def in_turn():
        with torch.cuda.stream(a):
            for token in new[1:]:
                for l, x in enumerate(token):
                    two[0].decode_step(l, *x, *two[1:])

    def own_predecessor():
        with torch.cuda.stream(a):
            two[0].decode_step(0, *new[1][0], *two[1:])
        b.wait_stream(a)
        with torch.cuda.stream(b):
            two[0].decode_step(1, *new[1][1], *two[1:])
        with torch.cuda.stream(a):
            two[0].decode_step(0, *new[2][0], *two[1:])

    graph, types, ok = capture(rt, [a, b], own_predecessor)          # never launched
    assert types and all(t == 0 for t in types)
    ok(rt.cudaGraphDestroy(graph))
    graph, types, ok = capture(rt, [a], in_turn)
    assert len(types) == 5 and all(t == 1 for t in types)
    run, = ok(rt.cudaGraphInstantiate(graph, 0))
    ok(rt.cudaGraphLaunch(run, a.cuda_stream))
    torch.cuda.synchronize()
    assert_same_decode_state(w, one, two)
    ok(rt.cudaGraphExecDestroy(run))
    ok(rt.cudaGraphDestroy(graph))


def cluster_widths(graph):
    """The cluster dimension of every kernel of a captured graph."""
    lib, n = ctypes.CDLL("libcudart.so.12"), ctypes.c_size_t(0)
    handle = ctypes.c_void_p(int(graph))
    assert lib.cudaGraphGetNodes(handle, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert lib.cudaGraphGetNodes(handle, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        val = (ctypes.c_uint32 * 16)()
        assert lib.cudaGraphKernelNodeGetAttribute(ctypes.c_void_p(node), 4, val) == 0      # cluster dimension
        out.append(val[0])
    return out


@pytest.mark.parametrize("bound", [None, 16, 8, 4, 1])
def test_cluster_width_follows_its_bound(monkeypatch, bound):
    """Heads that the decode step spreads over 16 CTAs, and a selection that does: with a lower bound, as on a
    device that holds no cluster of 16, the launches stay within it and the results are the same."""
    rt = pytest.importorskip("cuda.bindings.runtime")
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=4, n_kv_heads=2, seq_lens=(8000,), total_budget=4500)
    (one, two), new = decode_pair(w, tokens=2)
    vals = torch.randn(2, 70001, generator=torch.Generator().manual_seed(3)).cuda()
    want = binding.select_positions_static(vals, 900)
    for token in new:
        one[0].decode_step(0, *token[0], *one[1:])
    if bound is not None:
        monkeypatch.setenv("CAKE_MAX_CLUSTER", str(bound))
    out = torch.empty_like(want)
    two[0].decode_step(0, *new[0][0], *two[1:])
    torch.cuda.synchronize()
    st = torch.cuda.Stream()

    def body():
        with torch.cuda.stream(st):
            two[0].decode_step(0, *new[1][0], *two[1:])
            binding.select_positions_static(vals, 900, out=out)

    graph, _, ok = capture(rt, [st], body)
    assert sorted(cluster_widths(graph)) == [bound or 16, bound or 16]
    run, = ok(rt.cudaGraphInstantiate(graph, 0))
    ok(rt.cudaGraphLaunch(run, st.cuda_stream))
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    got, ref = ([x.clone() for x in c[0].decode_get_state(0, 0, 4500)] for c in (two, one))
    assert torch.equal(got[0], ref[0]) and torch.equal(got[2], ref[2])
    assert torch.allclose(got[1], ref[1], rtol=RTOL, atol=1e-12)
    for c in (one, two):
        assert c[0].status() == 0
        c[0].destroy()
    ok(rt.cudaGraphExecDestroy(run))
    ok(rt.cudaGraphDestroy(graph))

"""Scores where the passes can go wrong: prompts whose window starts at every place in a chunk of 16 keys, a tile of
128 and a CTA's share, and rows whose largest logit lies far above those of their first keys (the running reference
moves up, or the tile is taken again from its maxima).  Indicators and preferences against the float64 oracle
with the tolerance of the parity tests (1e-3 relative: bf16 inputs, fp32 accumulation)."""
import numpy as np
import pytest
import torch

from oracle import cake_oracle as O
from paper_2503_12491_b200 import binding, harness, synth

pytestmark = pytest.mark.gpu

RTOL = 1e-3


def check(w, qs, ks):
    cake = harness.cake_for(w)
    cake.begin(w.cu_seqlens)
    cake.score_layer(0, qs[0], ks[0])
    ind = cake.get_indicators(0).cpu().numpy()
    P = cake.get_preferences()[2].cpu().numpy()
    cu = w.cu_seqlens
    for r, N in enumerate(w.seq_lens):
        ref = O.score_layer(qs[0][r].float().cpu().numpy().astype(np.float64),
                            ks[0][:, cu[r]:cu[r + 1]].float().cpu().numpy().astype(np.float64),
                            gamma=w.gamma, pool_kernel=w.pool_kernel)
        got, want = ind[:, cu[r]:cu[r] + N - w.window], ref["indicator"]
        assert (np.abs(got - want) <= RTOL * np.abs(want) + 1e-30).all(), (r, N)
        assert abs(P[r, 0] - ref["P"]) <= RTOL * abs(ref["P"]) + 1e-30
    assert cake.status() == 0
    cake.destroy()


@pytest.mark.parametrize("hq,hkv,window,d", [(8, 2, 32, 128), (2, 2, 32, 64), (4, 2, 32, 128), (8, 1, 16, 64)])
@pytest.mark.parametrize("first", [33, 128, 143, 160, 239, 1024])
def test_windows_at_every_place_of_a_chunk(hq, hkv, window, d, first):
    lens = tuple(first + i for i in range(0, 18, 1 if first < 200 else 5))
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, window=window, seq_lens=lens,
                     total_budget=window + 20)
    qs, ks, _ = harness.device_inputs(w)
    check(w, qs, ks)


@pytest.mark.parametrize("jump", [8.0, 45.0, 65.0, 90.0, 300.0])
@pytest.mark.parametrize("hq,hkv", [(8, 2), (2, 2)])
def test_a_logit_far_above_the_first_keys(hq, hkv, jump):
    """Window queries and one key share a direction: that key's logits are `jump` nats above the others, which
    are of the order of one, for the rows of even index; it lies in a later tile of its CTA's share."""
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=hq, n_kv_heads=hkv, seq_lens=(20000, 700), total_budget=60)
    gen = torch.Generator().manual_seed(7)
    d = w.head_dim
    q = torch.randn(2, hq, w.window, d, generator=gen)
    k = torch.randn(hkv, w.total_tokens, d, generator=gen)
    q[..., 0] = 0.0
    q[:, :, ::2, 0] = 4.0
    k[..., 0] = 0.0
    k[:, [130, 390, 517, 9001, 15555, 20000 + 400], 0] = jump * d ** 0.5 / 4.0
    check(w, [q.bfloat16().cuda()], [k.bfloat16().cuda()])


@pytest.mark.parametrize("hq,hkv,window", [(2, 2, 3), (2, 2, 33), (4, 2, 31), (4, 2, 33), (6, 2, 13), (8, 2, 17), (16, 2, 7), (16, 2, 9)])
def test_fp32_windows_around_a_batch_of_rows(hq, hkv, window):
    """The column pass of fp32 inputs takes a quarter of the window rows in batches of 2 to 8.  Three layers in a row,
    on other inputs each: a layer's kernels start while the ones before them end."""
    w = synth.scaled(synth.workload(1), n_layers=3, n_q_heads=hq, n_kv_heads=hkv, window=window, seq_lens=(window + 1, 150, 700),
                     total_budget=3 * (window + 20))
    qs, ks, _ = harness.device_inputs(w)
    cake = harness.cake_for(w)
    cake.begin(w.cu_seqlens)
    ind = []
    for l in range(w.n_layers):
        cake.score_layer(l, qs[l], ks[l])
        ind.append(cake.get_indicators(l))
        cake.allocate(l)
        cake.evict(l)
    P, cu = cake.get_preferences()[2].cpu().numpy(), w.cu_seqlens
    for l in range(w.n_layers):
        for r, N in enumerate(w.seq_lens):
            ref = O.score_layer(qs[l][r].cpu().numpy().astype(np.float64), ks[l][:, cu[r]:cu[r + 1]].cpu().numpy().astype(np.float64),
                                gamma=w.gamma, pool_kernel=w.pool_kernel)
            got, want = ind[l].cpu().numpy()[:, cu[r]:cu[r] + N - w.window], ref["indicator"]
            assert (np.abs(got - want) <= RTOL * np.abs(want) + 1e-30).all(), (l, r)
            assert abs(P[r, l] - ref["P"]) <= RTOL * abs(ref["P"]) + 1e-30
    assert cake.status() == 0
    cake.destroy()


@pytest.mark.parametrize("hq,hkv,window,dtype", [(8, 2, 32, "bf16"), (2, 2, 32, "bf16"), (4, 2, 32, "bf16"), (8, 2, 32, "fp32")])
@pytest.mark.parametrize("tokens", [300, 700, 6100])
def test_infinite_logits_are_reported(hq, hkv, window, dtype, tokens):
    """A channel of some keys is infinite (an overflow): a run of 16 or 40 keys at the start of the prompt or of every
    tile, seen by queries of one sign or of both, so that a row's first logits of a tile are all -inf while its
    neighbours' are finite or inf.  The status says so, and the next batch of the context is not touched by it.  One
    request, at 6100 tokens with several tiles per warp, and two."""
    lens = (tokens,) if tokens != 700 else (tokens, 450)
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=hq, n_kv_heads=hkv, window=window, seq_lens=lens,
                     total_budget=window + 20, dtype=dtype)
    if tokens == 6100:                               # more pairs than the device has SMs for: several tiles per CTA
        w = synth.scaled(w, seq_lens=(tokens,) * 24)
    (q0,), (k0,), _ = harness.device_inputs(w)
    q0[..., 0] = q0[..., 0].abs() + 0.5
    cake = harness.cake_for(w)

    def score(q, k):
        cake.begin(w.cu_seqlens)
        cake.score_layer(0, q, k)
        out = cake.get_indicators(0), *cake.get_preferences()
        return cake.status(), out

    status, fresh = score(q0, k0)
    assert status == 0
    for sign in ("one", "both"):
        q = q0.clone()
        if sign == "both":
            q[:, :, ::2, 0] *= -1
        for run in (16, 40):
            for where in ("start", "tiles"):
                for value in (float("inf"), float("-inf")):
                    k = k0.clone()
                    for r, N in enumerate(w.seq_lens):
                        rows = torch.arange(N - window, device="cuda")
                        rows = rows[(rows % 128 if where == "tiles" else rows) < run] + w.cu_seqlens[r]
                        k[:, rows, 0] = value
                    status, _ = score(q, k)
                    assert status == binding.CAKE_ERR_NONFINITE, (sign, run, where, value)
                    status, again = score(q0, k0)
                    assert status == 0 and all(torch.equal(a, b) for a, b in zip(fresh, again))
    cake.destroy()


@pytest.mark.parametrize("hq,hkv", [(8, 2), (2, 2), (4, 2)])
@pytest.mark.parametrize("first", [16, 128, 144, 149, 2096])
def test_nan_in_the_window_is_reported(hq, hkv, first):
    """Window keys that are NaN: the rows of a chunk at the end of the prompt may see nothing but NaN in it."""
    w = synth.scaled(synth.workload(3), n_layers=1, n_q_heads=hq, n_kv_heads=hkv, seq_lens=(first + 32,), total_budget=32 + 5)
    (q,), (k0,), _ = harness.device_inputs(w)
    cake = harness.cake_for(w)
    for lo, hi in ((0, 32), (0, 16), (16, 32), (31, 32), (0, 0)):
        k = k0.clone()
        k[:, first + lo:first + hi] = float("nan")
        cake.begin(w.cu_seqlens)
        cake.score_layer(0, q, k)
        assert cake.status() == (binding.CAKE_ERR_NONFINITE if hi > lo else 0), (lo, hi)
    cake.destroy()

"""Which positions a budget keeps, where the selection can go wrong: rows that start at every 16-byte offset
and end around the groups of 8 and 32 values, threshold buckets with more values than the list in shared
memory holds, many equal values at the cut, thresholds below zero, infinite and lowest values.
Positions are whole numbers and are compared exactly with the oracle's TopK on the same values."""
import numpy as np
import pytest
import torch

from oracle import cake_oracle as O
from paper_2503_12491_b200 import harness, synth

pytestmark = pytest.mark.gpu

WINDOW = 2


def values(kind, n, rng):
    x = rng.normal(size=n).astype(np.float32)
    if kind == "spread":
        return np.exp(x)
    if kind == "one bucket":                         # distinct values with the same leading bits
        return (1.0 + rng.permutation(n) / (16.0 * n)).astype(np.float32)
    if kind == "all equal":
        return np.full(n, 0.25, dtype=np.float32)
    if kind == "ties":                               # a third of the values equal, around the cut
        return np.where(rng.random(n) < 0.33, np.float32(1.0), np.exp(x))
    if kind == "negative":
        return -np.exp(x)
    if kind == "bucket edges":                       # around the powers of two where fine buckets begin and end
        return (np.exp2(rng.choice([-30, -28, -27, -26, 4, 5, 6], size=n)) * (1 + rng.integers(-2, 3, size=n) / 64)).astype(np.float32)
    x[rng.random(n) < 0.1] = np.inf                  # "extremes"
    x[rng.random(n) < 0.3] = np.finfo(np.float32).min
    return x


@pytest.mark.parametrize("lens", [(901, 902, 903, 904, 31, 33), (3, 34, 35, 4090, 4103), (40007,), (131072,)])
@pytest.mark.parametrize("kind", ["spread", "one bucket", "all equal", "ties", "negative", "extremes"])
def test_positions_of_a_budget(kind, lens):
    w = synth.scaled(synth.workload(1), n_layers=1, n_q_heads=3, n_kv_heads=3, window=WINDOW, seq_lens=lens,
                     total_budget=WINDOW + max(lens) // 7 + 1)
    rng = np.random.default_rng(len(kind) + max(lens))
    ind = np.zeros((w.n_kv_heads, w.total_tokens), dtype=np.float32)
    cu = w.cu_seqlens
    for g in range(w.n_kv_heads):
        for r, N in enumerate(lens):
            ind[g, cu[r]:cu[r] + N - WINDOW] = values(kind, N - WINDOW, rng)
    cake = harness.cake_for(w)
    cake.begin(cu)
    cake.set_preferences(torch.ones(len(lens), 1, dtype=torch.float64, device="cuda"))
    cake.set_indicators(0, torch.from_numpy(ind).cuda())
    cake.allocate(0)
    cake.evict(0)
    budgets = cake.get_budgets().cpu().numpy()
    for r, N in enumerate(lens):
        n, b = N - WINDOW, int(budgets[r, 0])
        got = cake.get_positions(r, 0, b).cpu().numpy()
        for g in range(w.n_kv_heads):
            want = np.concatenate([O.topk_keep(ind[g, cu[r]:cu[r] + n].astype(np.float64), b - WINDOW), np.arange(n, N)])
            assert np.array_equal(got[g], want), (r, g)
    assert cake.status() == 0
    cake.destroy()


@pytest.mark.parametrize("kind", ["bucket edges", "spread", "one bucket", "all equal"])
@pytest.mark.parametrize("lens", [(33, 70_001, 517, 131_072), (32_739, 32_770), (16_418,), (8_225, 3)])
def test_lists_that_several_ctas_share(kind, lens):
    """Few lists are spread over clusters: runs of values that end inside a word, CTAs without any, candidates of one
    bucket in all of them, and buckets on either side of the range with finer ones."""
    test_positions_of_a_budget(kind, lens)


@pytest.mark.parametrize("reader", ["compact", "int4", "positions", "budgets"])
@pytest.mark.parametrize("streams", ["one", "two"])
def test_budgets_are_read_before_they_are_written_again(reader, streams):
    """The buffer of a stage's budgets is written again two stages later, on the internal stream: results handed out
    behind a long wait of the caller's stream are still those of their stage, also where another stream reads after it."""
    w = synth.scaled(synth.workload(1), n_layers=3, n_q_heads=2, n_kv_heads=2, window=WINDOW, seq_lens=(3000,), total_budget=900)
    gen = torch.Generator(device="cuda").manual_seed(3)
    k = [torch.randn(2, 3000, w.head_dim, generator=gen, device="cuda") for _ in range(3)]
    x = torch.rand(2, 3000, generator=gen, device="cuda")
    cake = harness.cake_for(w)

    def read():
        if reader == "compact":
            rows = cake.packed_rows_bound()
            out = cake.compact(k, k, layer_hi=1, k_out=torch.zeros(rows, w.head_dim, device="cuda"),
                               v_out=torch.zeros(rows, w.head_dim, device="cuda"), positions=torch.zeros(rows, dtype=torch.int32, device="cuda"))
            return list(out)
        if reader == "budgets":
            return [cake.get_budgets()]
        return [cake.get_positions(0, 0, 896)]

    def run(wait):
        cake.begin(w.cu_seqlens)
        cake.set_preferences(torch.ones(1, 3, dtype=torch.float64, device="cuda"))
        for l in range(3 if reader == "int4" else 1):
            cake.set_indicators(l, x)
            cake.allocate(l)
            cake.evict(l)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        with torch.cuda.stream(side if streams == "two" else torch.cuda.current_stream()):
            if wait:
                torch.cuda._sleep(20_000_000)        # about ten milliseconds
            if reader == "int4":
                out = cake.compact_int4(k, k)
                out = [out["row_offsets"], out["positions"][:1800], out["k_codes"][:1800]]
            else:
                out = read()
        if streams == "two":
            cake.get_budgets()
        if wait:
            for stage in (0,) if reader == "int4" else (1, 2):      # (INT4 compaction has read the budgets of stage 2)
                cake.allocate(stage)
        torch.cuda.synchronize()
        return out

    want, got = run(False), run(True)
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    assert cake.status() == 0
    cake.destroy()


@pytest.mark.parametrize("lens", [(1_600_003,), (1_600_003, 3001, 90_007), (517, 1_580_000, 1_600_001)])
@pytest.mark.parametrize("kind", ["spread", "one bucket", "ties"])
@pytest.mark.parametrize("cluster", ["8", "1"])
def test_prompts_beyond_the_shared_memory_bitmap(kind, lens, cluster, monkeypatch):
    """Requests of more than 1.2 M tokens, alone and beside short ones: a CTA's bitmap does not fit its shared memory
    (with one CTA per list) and lies in global scratch, which is sized by the sum of the tokens."""
    monkeypatch.setenv("CAKE_MAX_CLUSTER", cluster)
    w = synth.scaled(synth.workload(1), n_layers=1, n_q_heads=1, n_kv_heads=1, window=WINDOW, seq_lens=lens,
                     total_budget=WINDOW + 100_001, dtype="bf16")
    rng = np.random.default_rng(len(kind) + len(lens))
    cu = w.cu_seqlens
    ind = np.zeros((1, w.total_tokens), dtype=np.float32)
    for r, N in enumerate(lens):
        ind[0, cu[r]:cu[r] + N - WINDOW] = values(kind, N - WINDOW, rng)
    cake = harness.cake_for(w)
    cake.begin(cu)
    cake.set_preferences(torch.ones(len(lens), 1, dtype=torch.float64, device="cuda"))
    cake.set_indicators(0, torch.from_numpy(ind).cuda())
    cake.allocate(0)
    cake.evict(0)
    k = torch.zeros(1, w.total_tokens, w.head_dim, dtype=torch.bfloat16, device="cuda")
    _, _, off, pos = cake.compact([k], [k])
    off, pos = off.tolist(), pos.cpu().numpy()
    for r, N in enumerate(lens):
        n = N - WINDOW
        b = min(n, 100_001)
        want = np.concatenate([O.topk_keep(ind[0, cu[r]:cu[r] + n].astype(np.float64), b), np.arange(n, N)])
        assert np.array_equal(pos[off[r]:off[r + 1]], want), r
        assert np.array_equal(cake.get_positions(r, 0, b + WINDOW).cpu().numpy()[0], want), r
    assert cake.status() == 0
    cake.destroy()

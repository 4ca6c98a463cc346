"""Grouping of an append by id range, counted and placed in tiles of 1 024 rows for up to 64 ranges and small enough appends, sorted beyond; and the pieces
of a launch, 64 of them in the launch itself, a table in memory beyond: either side of every limit, several tiles, ranges that get nothing, ids
that are refused.  Runs against the oracle's writer, bit for bit."""
import numpy as np
import pytest

from oracle import run_store as rs
from test_gpu_runs import compare_with_oracle, rows_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,R,cuts", [
    (1, 900, (1_023, 2_047, 5_000)), (2, 4_000, (1, 1_025, 9_000)), (16, 100, (1_024, 3_073, 20_000)), (63, 50, (2_048, 2_049, 70_000)),
    (64, 40, (100, 1_124, 70_000)), (65, 40, (1_024, 30_000)), (64, 3_000, (300_000,)), (300, 7, (5_000, 5_001)),
])
def test_sizes(P, R, cuts):
    import torch
    import paper_2607_17374_b200 as tb
    dev = torch.device("cuda:0")
    V, width = cuts[-1] + 137, 4
    rng = np.random.default_rng(P + V)
    order = rng.permutation(V).astype(np.int64)
    order[:700] = np.sort(order[:700])           # some of it in order, and much of one range in a row
    runs = tb.Runs(V, width, P, R, store_kind=tb.RUNS_DEVICE)
    w = rs.RunWriter(V, P, R, width)
    for _ in range(2):
        for a, b in zip((0,) + cuts, cuts + (V,)):
            ids = order[a:b]
            rows = rows_for(ids, width)
            w.append(ids, rows)
            runs.append(torch.from_numpy(ids.copy()).to(dev), torch.from_numpy(rows).to(dev), width, b - a)
        runs.flush()
        w.flush()
        compare_with_oracle(runs, w, width)
        dense = rows_for(np.arange(V), width)
        for s, e in ((0, V), (1, 2), (V // 3, V // 2 + 1)):
            out = torch.full((e - s, width), -1.0, device=dev)
            runs.read_chunk(s, e, out, width)
            assert np.array_equal(out.cpu().numpy(), dense[s:e])
        runs.reset()
        w = rs.RunWriter(V, P, R, width)
    runs.destroy()


@pytest.mark.parametrize("P", [5, 64, 65])
@pytest.mark.parametrize("bad", [-1, 4_000, 2 ** 40])
def test_ids_that_are_no_vertices(P, bad):
    """Refused, whatever path; the rows that came before are still there and the next append goes through."""
    import torch
    import paper_2607_17374_b200 as tb
    V, width = 4_000, 4
    runs = tb.Runs(V, width, P, 64, store_kind=tb.RUNS_DEVICE)
    ids = np.arange(V, dtype=np.int64)

    def append(part):
        runs.append(torch.from_numpy(part.copy()).cuda(), torch.from_numpy(rows_for(np.clip(part, 0, V - 1), width)).cuda(), width, len(part))
    append(ids[:1_500])
    wrong = ids[1_500:4_000].copy()
    wrong[1_777] = bad
    with pytest.raises(tb.TaurusError):
        append(wrong)
    append(ids[1_500:])
    runs.flush()
    out = torch.empty(V, width, device="cuda")
    runs.read_chunk(0, V, out, width)
    assert np.array_equal(out.cpu().numpy(), rows_for(ids, width))
    runs.destroy()

"""The cost model's report: the library's own kernel is timed as itself, not as
the table tile that it is named after."""
import pytest

from paper_2110_14340_gb300 import costmodel, jacc


def test_own_kernel_regret_is_its_own_time_against_the_best_tile():
    inf = float("inf")
    ms = [4.0, 2.0, 3.0, inf] + [8.0] * 20
    rows = [dict(stencil=7, dtype=32, side=64, ms=ms, valid=[m < inf for m in ms], own_ms=own) for own in (1.0, 2.0, 3.0)]
    assert costmodel.own_regret(rows) == [-0.5, 0.0, 0.5]
    assert costmodel.own_regret([{k: v for k, v in rows[0].items() if k != "own_ms"}]) == []


@pytest.mark.gpu
def test_collection_times_the_own_kernel():
    # 27-point FP32 64^3: the own kernel takes half of the fastest tile's time
    bufs = costmodel.Buffers(64 ** 3, dtypes=(32,))
    row, = costmodel.collect([(27, 32, 64)], bufs)
    assert 0.0 < row["own_ms"] < min(row["ms"])
    assert costmodel.own_regret([row])[0] < 0.0
    jacc.autotune_forget()

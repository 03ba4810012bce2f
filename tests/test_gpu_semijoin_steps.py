"""Semi-join counts where warps' steps of 256 rows and the 32-row counts end,
one to four dimensions, each held in shared memory or probed in place."""
import numpy as np
import pytest
import torch

from tests._helpers import as_columns

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 255, 256, 257, 1023, 1025, 8_191, 300_001, 1_300_000])
@pytest.mark.parametrize("dims", [(40,), (1_000_003,), (1_000_003, 31), (0, 33, 5000), (900_000, 64, 2, 800_001)])
def test_steps(rows, dims):
    from paper_1901_01488_gb300 import esc
    rng = np.random.default_rng(rows + len(dims))
    keys, marks, words = {}, [], []
    for d, n in enumerate(dims):
        k = rng.integers(-3, n + 5, rows).astype(np.int32)
        k[: min(rows, 3)] = [np.iinfo(np.int32).min, np.iinfo(np.int32).max, max(0, n - 1)][: min(rows, 3)]
        keys[f"fk{d}"] = k
        bits = rng.random((n + 31) // 32 * 32) < 0.4      # bits past the last row may be set: they never count
        ok = (k >= 0) & (k < n)
        marks.append(ok & bits[np.where(ok, k, 0)] if n else ok)
        w = np.packbits(bits, bitorder="little").view(np.int32) if n else np.zeros(1, np.int32)
        words.append(torch.from_numpy(w.copy()).cuda())
    t = esc.Table(as_columns(keys, "cuda"), rows)
    got = esc.esc_semijoin_counts(t.handle, list(keys), words, list(dims))
    for s in range(1 << len(dims)):
        m = np.ones(rows, bool)
        for d in range(len(dims)):
            if s >> d & 1:
                m &= marks[d]
        assert got[s] == int(m.sum()), s

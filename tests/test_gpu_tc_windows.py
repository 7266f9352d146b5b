"""Accumulation windows of the tensor-core contraction over window lengths that leave a block's short window 1 to 4
chunks, and set lengths below the slot count (which are raised above it), against the default window's result (its own
test compares that with the oracle); a drain that came early would add a whole window twice (a relative error of one
window in a block's chunks, 1e-2 and more here)."""
import numpy as np
import pytest

import fieldgen

torch = pytest.importorskip("torch")
import paper_1904_11055_gb300 as ps  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,order,nshell", [(64, 3, 16), (64, 4, 10), (48, 3, 12), (64, 2, 12)])
def test_short_last_windows(N, order, nshell, monkeypatch):
    e = fieldgen.unit_edges(nshell)
    d = torch.from_numpy(fieldgen.field("lognormal", N, 81, np.float32)).cuda()
    ref, scale = None, None
    for window in (None, 1, 2, 3, 4, 5, 6, 7, 9, 11, 13, 16, 27, 64):
        if window is None:
            monkeypatch.delenv("POLY_TC_WINDOW", raising=False)
        else:
            monkeypatch.setenv("POLY_TC_WINDOW", str(window))
        plan = ps.Plan(N, 500.0, order, e, "split_bf16")
        B, s = plan.estimate(d, scale=True)
        plan.sync()
        if ref is None:
            ref, scale = B, s * (500.0 ** 3) ** (order - 1) / float(N ** 3) ** order
        # both results lie within the split-BF16 bar (1e-5 of the scale) of the exact one
        assert float(((B - ref).abs() / scale).max()) <= 2e-5, window
        plan.close()

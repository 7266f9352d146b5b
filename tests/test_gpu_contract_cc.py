"""The CUDA-core contraction's blocks of bins at their edges, against the FP64 oracle.

A task covers one run of consecutive shells per leg; these cases have fewer shells than a run, shell counts
that are no multiple of one, single-task plans (several warps share a task), every order, and the sums of
absolute products (the error scale), whose kernel takes the same blocks."""
import numpy as np
import pytest

import fieldgen
import oracle

torch = pytest.importorskip("torch")
import paper_1904_11055_gb300 as ps  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp64": 1e-12}  # of sum |prod D|: FP32 products and partial sums (2^-24 each), FP64


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("N,order,nshell,flags", [
    (16, 2, 1, 0), (16, 3, 1, 0), (24, 3, 2, 0), (16, 4, 3, 0), (24, 5, 4, 0), (24, 6, 3, 0),
    (48, 2, 19, ps.POLY_BINS_ALL_SORTED), (32, 3, 9, ps.POLY_BINS_ALL_SORTED), (48, 3, 13, 0), (32, 4, 7, 0)])
def test_blocks_match_oracle(prec, N, order, nshell, flags):
    e = fieldgen.unit_edges(nshell)
    d = fieldgen.field("lognormal", N, 90 + nshell, np.float32)
    plan = ps.Plan(N, 500.0, order, e, prec, flags)
    x = torch.from_numpy(d).cuda().to(plan.real_dtype)
    B, scale = (t.cpu().numpy() for t in plan.estimate(x, scale=True))
    ref = oracle.estimate(d.astype(np.float64), 500.0, e, order, bins=plan.bins)
    assert np.array_equal(plan.counts, ref["counts"])
    some = plan.counts > 0
    c = (500.0 ** 3) ** (order - 1) / float(N ** 3) ** order
    assert np.all(B[~some] == 0)
    assert np.max(np.abs(B - ref["B"])[some] / (c * ref["scale"][some])) <= TOL[prec]
    assert np.max(np.abs(scale - ref["scale"])[some] / ref["scale"][some]) <= TOL[prec]
    plan.close()


def test_fp32_lanes_are_added_without_rounding():
    """FP32 sums are rounded within a lane only (some hundred cells).  Three waves of a quarter of the grid's frequency
    with 11-bit amplitudes make every cell's square an integer of at most 23 bits times a power of two, which a lane's
    few cells of this plan add without rounding; the lanes' sums together take 30 bits and more."""
    N, L = 64, 500.0
    c = torch.cos(0.5 * np.pi * torch.arange(N, dtype=torch.float64)).round()
    d = 947 * c[:, None, None] + 613 * c[None, :, None] + 311 * c[None, None, :]
    plan = ps.Plan(N, L, 2, np.array([15.5, 16.5]), "fp32")
    B, scale = plan.estimate(d.float().cuda(), scale=True)
    S = float((d ** 2).sum())  # sum of D^2 over N^6, an integer below 2^53
    want = L ** 3 * S / (float(N) ** 3 * float(plan.counts[0]))
    assert float(B[0]) == pytest.approx(want, rel=1e-12)
    assert float(scale[0]) * L ** 3 / float(N) ** 6 == pytest.approx(want, rel=1e-12)
    plan.close()

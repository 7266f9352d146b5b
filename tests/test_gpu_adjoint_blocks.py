"""The CUDA-core adjoint's blocks of output shells (eight in FP32, four in FP64) at their edges, against the FP64 oracle's gradient:
one shell, a partial block, exactly one block or two, one shell more, and several blocks, in every order it serves
(orders 2 and 4 of split-BF16 plans run here too)."""
import numpy as np
import pytest

import fieldgen
import oracle

torch = pytest.importorskip("torch")
import paper_1904_11055_gb300 as ps  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-5, "split_bf16": 2e-5, "fp64": 1e-10}  # of the largest component, as the other adjoint tests


@pytest.mark.parametrize("N,order,nshell,prec,flags", [
    (16, 3, 1, "fp32", 0), (32, 3, 7, "fp32", 0), (32, 3, 8, "fp64", 0), (32, 3, 9, "fp32", 0), (64, 3, 19, "fp32", 0),
    (32, 2, 11, "fp32", ps.POLY_BINS_ALL_SORTED), (24, 2, 8, "fp64", 0), (32, 4, 7, "fp32", 0), (24, 4, 5, "split_bf16", 0),
    (48, 4, 9, "fp64", 0), (32, 3, 9, "fp64", ps.POLY_BINS_ALL_SORTED)])
def test_gradient_blocks_match_oracle(N, order, nshell, prec, flags):
    e = fieldgen.unit_edges(nshell)
    d = fieldgen.field("lognormal", N, 70 + nshell, np.float32)
    plan = ps.Plan(N, 500.0, order, e, prec, flags)
    w = np.random.default_rng(nshell).standard_normal(plan.nbins) * (plan.counts > 0)
    x = torch.from_numpy(d).cuda().to(plan.real_dtype)
    for _ in range(2):  # a second call finds the first one's weights and tables
        g = plan.backward(x, torch.from_numpy(w).cuda())
    plan.sync()
    some = plan.counts > 0
    ref = oracle.gradient(d.astype(np.float64), 500.0, e, order, plan.bins[some], plan.counts[some], w[some])
    assert np.abs(g.double().cpu().numpy() - ref).max() <= TOL[prec] * np.abs(ref).max()
    plan.close()

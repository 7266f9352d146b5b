"""The CUDA-core adjoint's blocks of output shells (eight in FP32, four in FP64) at their edges, against the FP64 oracle's gradient:
one shell, a partial block, exactly one block or two, one shell more, and several blocks, in every order it serves
(orders 2 and 4 of split-BF16 plans run here too).  And the tensor-core adjoint's chunks of 8 by 8 shells and
16-column blocks: partial ones, one chunk, an odd and an even count of them, several accumulation segments, the
most shells of the pair form, and one more (narrow shells, some of them empty), which takes the other form."""
import numpy as np
import pytest

import fieldgen
import oracle

torch = pytest.importorskip("torch")
import paper_1904_11055_gb300 as ps  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-5, "split_bf16": 2e-5, "fp64": 1e-10}  # of the largest component, as the other adjoint tests


def check(N, order, edges, prec, flags, seed):
    d = fieldgen.field("lognormal", N, seed, np.float32)
    plan = ps.Plan(N, 500.0, order, edges, prec, flags)
    w = np.random.default_rng(seed).standard_normal(plan.nbins) * (plan.counts > 0)
    x = torch.from_numpy(d).cuda().to(plan.real_dtype)
    for _ in range(2):  # a second call finds the first one's weights and tables
        g = plan.backward(x, torch.from_numpy(w).cuda())
    plan.sync()
    some = plan.counts > 0
    ref = oracle.gradient(d.astype(np.float64), 500.0, edges, order, plan.bins[some], plan.counts[some], w[some])
    assert np.abs(g.double().cpu().numpy() - ref).max() <= TOL[prec] * np.abs(ref).max()
    plan.close()


@pytest.mark.parametrize("N,nshell,width", [(16, 1, 1.0), (16, 4, 1.0), (32, 5, 1.0), (32, 9, 1.0), (48, 13, 1.0), (64, 16, 1.0),
                                            (64, 17, 1.0), (32, 33, 0.3), (32, 64, 0.15), (32, 65, 0.15)])
def test_pair_gradient_matches_oracle(N, nshell, width):
    check(N, 3, fieldgen.unit_edges(nshell, width), "split_bf16", 0, 170 + nshell)


@pytest.mark.parametrize("N,order,nshell,prec,flags", [
    (16, 3, 1, "fp32", 0), (32, 3, 7, "fp32", 0), (32, 3, 8, "fp64", 0), (32, 3, 9, "fp32", 0), (64, 3, 19, "fp32", 0),
    (32, 2, 11, "fp32", ps.POLY_BINS_ALL_SORTED), (24, 2, 8, "fp64", 0), (32, 4, 7, "fp32", 0), (24, 4, 5, "split_bf16", 0),
    (48, 4, 9, "fp64", 0), (32, 3, 9, "fp64", ps.POLY_BINS_ALL_SORTED)])
def test_gradient_blocks_match_oracle(N, order, nshell, prec, flags):
    check(N, order, fieldgen.unit_edges(nshell), prec, flags, 70 + nshell)


@pytest.mark.parametrize("nshell", [20, 40, 52, 64])
def test_pair_gradient_error_against_64_bits(nshell):
    """The pairs' errors stay below those of the form over columns (m, j), which is what runs beyond 64 shells (2.8e-6 of
    the 2-norm with normal weights, 2.6e-6 to 3.2e-6 with weights over the bins' expected scatter).  Bounds: products
    split into bf16 hi + lo leave 2^-18 of each on average at random, below 5e-7 of the sum; then the tensor core's
    truncation, 2^-25 of the running sum for each of a segment's 96 accumulations, 2.9e-6 if all of them fell on the
    full sum.  With normal weights the last chunk holds nearly all of the sum, and 16 accumulations, 4.8e-7."""
    N = 128 if nshell <= 40 else 256
    e = fieldgen.unit_edges(nshell)
    x = torch.from_numpy(fieldgen.field("lognormal", N, 6, np.float32)).cuda()
    p64, p = ps.Plan(N, 500.0, 3, e, "fp64"), ps.Plan(N, 500.0, 3, e, "split_bf16")
    k = p.bins.astype(np.float64)
    scatter = np.exp(0.5 * (2.5 * np.log(k) + (k / (N / 4)) ** 2)).prod(axis=1)
    for seed in (1, 2, 4):
        r = np.random.default_rng(seed).standard_normal(p.nbins) * (p.counts > 0)
        for w, bound in ((r, 1e-6), (r * scatter, 3.4e-6)):
            w = torch.from_numpy(w).cuda()
            ref, g = p64.backward(x.double(), w), p.backward(x, w)
            p64.sync(), p.sync()
            assert float((g.double() - ref).norm() / ref.norm()) <= bound
    p64.close(), p.close()

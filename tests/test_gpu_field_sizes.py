"""Shell fields at the grid sizes whose transforms have their own stages or plane blocks.

96 = 12 x 8 and 160 = 16 x 10 are transformed with prime-factor butterflies of length 12
and 10, and 64, 96 and 160 run the narrow shells in blocks of 4 or 9 warps; 48 and 256 share
neither.  Narrow shells take the small blocks, the last one (out to the Nyquist edge up to 160^3) the
large one; an odd number of row pairs leaves the last group of a warp partly empty.

The bound: a length-n transform in a type of unit roundoff u has an error below
u log2(n) (a small constant) times the root mean square of its output; two transforms of
N^3 points, and the peak of a field of white noise is at least its root mean square, so
8 u log2(N^3) of the shell's peak bounds both directions with room for the butterflies'
constants (radix 5 and 3 take about twice the operations of radix 2 per bit).
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1904_11055_gb300 as ps  # noqa: E402
from test_zz_shell_fields import grid_q2, library_fields, shell_mask  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("N", [48, 64, 96, 160, 256])
def test_fields_match_the_transform_of_the_masked_spectrum(N, prec):
    top = min((N - 1) // 2, 70)
    edges = np.array([1.0, 2.0, 4.5, 9.0, top // 2 + 0.5, float(top)])
    dt = torch.float32 if prec == "fp32" else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(N)
    d = torch.randn(N, N, N, generator=gen, device="cuda", dtype=dt)
    plan = ps.Plan(N, 100.0, 2, edges, prec)
    got = library_fields(plan, d)
    F = torch.fft.fftn(d.double())
    _, q2 = grid_q2(N)
    tol = 8 * math.log2(N**3) * (2.0**-24 if prec == "fp32" else 2.0**-53)
    for s in range(len(edges) - 1):
        ref = (torch.fft.ifftn(F * shell_mask(q2, edges, s)).real * N**3).cpu().numpy()
        err = np.abs(got[s] - ref).max() / np.abs(ref).max()
        assert err < tol, (s, err, tol)


@pytest.mark.parametrize("prec,ell", [("fp32", 0), ("split_bf16", 0), ("split_bf16", 2)])
@pytest.mark.parametrize("K", [88, 89, 120])
def test_planes_beyond_shared_memory(K, prec, ell):
    """Single-precision planes of 256^3 fit shared memory up to K = 88; from 89 on they go through a buffer.  The
    fields as above, the power spectrum against the mean of |delta_hat|^2, and the gradient by Euler's theorem,
    delta . dB = 2 B.  Bounds: FP32 sums of squares over 512 cells, then FP64, 1e-5; split-BF16, the tensor core
    truncates a growing sum at each of a window's 128 x 2 x 3 accumulations by up to 2^-24 of it."""
    N, edges = 256, np.array([1.0, 30.5, K - 4.5, K + 0.5])
    gen = torch.Generator(device="cuda").manual_seed(K)
    d = torch.randn(N, N, N, generator=gen, device="cuda", dtype=torch.float32)
    plan = ps.Plan(N, 100.0, 2, edges, prec, 0, ell)
    B = plan.estimate(d)
    plan.sync()
    F = torch.fft.fftn(d.double())
    f, q2 = grid_q2(N)
    w = (2 * ell + 1) * (1.5 * f[None, None, :] ** 2 / q2.clamp(min=1.0) - 0.5) if ell else torch.ones_like(q2)
    P = (F.abs() ** 2 * w, F.abs() ** 2 * w.abs())
    c = 100.0**3 / float(N) ** 6
    tol = 768 * 2.0**-24 if prec == "split_bf16" else 1e-5
    for s in range(3):
        m = shell_mask(q2, edges, s)
        assert abs(float(B[s]) - c * float(P[0][m].mean())) <= tol * c * float(P[1][m].mean())
    if ell:
        return
    got = library_fields(plan, d)
    for s in range(3):
        ref = (torch.fft.ifftn(F * shell_mask(q2, edges, s)).real * N**3).cpu().numpy()
        assert np.abs(got[s] - ref).max() / np.abs(ref).max() < 8 * math.log2(N**3) * 2.0**-24
    wt = torch.tensor([1.0, 0.5, 2.0], dtype=torch.float64, device="cuda")
    g = plan.backward(d, wt)
    plan.sync()
    assert float((g.double() * d.double()).sum()) == pytest.approx(2 * float((wt * B).sum()), rel=2 * tol)

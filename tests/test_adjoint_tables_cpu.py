"""The tables that the adjoint's kernels walk, on the host: the tensor-core form over pairs of shells (split-BF16 plans of
up to 64 shells) and the CUDA-core form (all others).  Each is walked as its kernel does for one cell with random
fields and weights, and the sums are compared with the entries' definition,
G_m = sum over entries e of m of w_e times the product of e's other fields."""
import ctypes

import numpy as np
import pytest

import fieldgen
import paper_1904_11055_gb300 as ps
from paper_1904_11055_gb300 import build as psbuild
from test_host_tables_cpu import adj_tables, check_at_tables


@pytest.fixture(scope="module")
def lib():
    psbuild.build()
    return ps.load_library()


def definition(t, order, nshell, D, w):
    m = np.repeat(np.arange(nshell), np.diff(t["moff"]))
    p = w.copy()
    for q in range(order - 1):
        p *= D[t["ent"][:, q]]
    return np.bincount(m, p, nshell)


def pair_tables(lib, N, edges):
    fn, P = lib.poly_diag_adj_pairs, ctypes.c_void_p
    fn.argtypes = [ctypes.c_int, P, ctypes.c_int, ctypes.c_uint, P, P, P]
    e, sizes = np.ascontiguousarray(edges, np.float64), np.zeros(4, np.int64)
    args = (N, e.ctypes.data, e.size - 1, 0, sizes.ctypes.data)
    assert fn(*args, None, None) == 0
    chunks, place = np.zeros((sizes[0], 8), np.int32), np.zeros((sizes[1], 2), np.int32)
    assert fn(*args, chunks.ctypes.data, place.ctypes.data) == 0
    return chunks, place, int(sizes[2]), int(sizes[3])


@pytest.mark.parametrize("N,nshell,width", [(32, 1, 1.0), (32, 4, 1.0), (32, 8, 1.0), (48, 9, 1.0), (64, 16, 1.0), (64, 17, 1.0),
                                            (128, 32, 1.0), (128, 33, 1.0), (160, 48, 1.0), (160, 49, 1.0), (256, 64, 1.0),
                                            (32, 64, 0.15), (256, 5, 2.0)])
def test_pair_tables(lib, N, nshell, width):
    edges = fieldgen.unit_edges(nshell, width)
    t = adj_tables(lib, N, 3, edges, "split_bf16")
    chunks, place, nbytes, smem = pair_tables(lib, N, edges)
    assert len(chunks) >= 3 and smem <= 227 * 1024  # every group of producers has a chunk of each tile
    rng = np.random.default_rng(nshell)
    D, w = rng.standard_normal(nshell), rng.standard_normal(len(place))
    stored = {}
    for (at, part), v in zip(place.tolist(), w):
        for k in range(3):  # three parts, at their own places
            assert (at + k * part) not in stored and 0 <= at + k * part < nbytes
            stored[at + k * part] = v if k == 0 else 0.0
    sums, acc, used, ends, starts = np.zeros(nshell + 16), None, 0, [], 0
    nblk = (nshell + 15) // 16 * 16
    for c, (jb, i0, n0, nn, off, first, last, _) in enumerate(chunks.tolist()):
        if first:
            assert acc is None and starts == len(ends) and nn == nblk and n0 == 0 and jb >= 0  # overwrites every column
            acc = np.zeros(nblk)
            starts += 1
        if jb >= 0:
            assert nn > 0 and nn % 16 == 0 and n0 % 16 == 0 and n0 + nn <= nblk and nn * 384 * 4 <= smem
            for n in range(nn):
                for k in range(64):
                    at = off + n // 8 * 1024 + k // 8 * 128 + n % 8 * 16 + k % 8 * 2
                    if at in stored:
                        used += 1
                        assert n0 + n < nshell and at + nn * 128 in stored and at + nn * 256 in stored  # where the kernel reads the other parts
                        acc[n0 + n] += stored[at] * D[i0 + k // 8] * D[jb + k % 8]
            assert off + nn * 384 <= nbytes
        else:
            assert nn == 0
        if last:
            sums[:nblk] += acc[:nblk] if nblk <= len(sums) else acc
            acc = None
            ends.append(c)
    assert acc is None and ends[-1] == len(chunks) - 1 and chunks[:len(ends), 7].tolist() == ends
    assert used == len(place)  # every weight was met once (its first part; the others lie in the next parts)
    ref = definition(t, 3, nshell, D, w)
    assert np.allclose(sums[:nshell], ref, rtol=0, atol=1e-9 * max(1.0, np.abs(ref).max()))


@pytest.mark.parametrize("N,nshell,width", [(256, 65, 1.0), (128, 70, 0.6), (256, 4, 1.0), (256, 3, 2.0)])
def test_other_plans_take_the_columns(lib, N, nshell, width):
    edges = fieldgen.unit_edges(nshell, width)
    assert len(pair_tables(lib, N, edges)[0]) == 0
    t = adj_tables(lib, N, 3, edges, "split_bf16")
    assert len(t["groups"]) > 0
    check_at_tables(t, nshell)


@pytest.mark.parametrize("N,order,nshell,width,prec", [
    (32, 3, 1, 1.0, "fp32"), (32, 3, 8, 1.0, "fp32"), (48, 3, 9, 1.0, "fp32"), (128, 3, 40, 1.0, "fp32"), (64, 3, 16, 1.0, "fp64"),
    (64, 3, 17, 1.0, "fp64"), (64, 2, 11, 1.0, "fp32"), (24, 2, 8, 1.0, "fp64"), (64, 4, 9, 1.5, "fp32"), (64, 4, 10, 1.5, "fp64"),
    (128, 4, 20, 1.5, "fp32")])
def test_block_tables(lib, N, order, nshell, width, prec):
    fn, P = lib.poly_diag_adj_blocks, ctypes.c_void_p
    fn.argtypes = [ctypes.c_int, ctypes.c_int, P, ctypes.c_int, ctypes.c_uint, ctypes.c_int, P, P, P, P]
    e, sizes = np.ascontiguousarray(fieldgen.unit_edges(nshell, width), np.float64), np.zeros(6, np.int64)
    args = (N, order, e.ctypes.data, nshell, 0, ps.PRECISIONS[prec], sizes.ctypes.data)
    assert fn(*args, None, None, None) == 0
    blocks, segs, place = np.zeros((sizes[0], 5), np.int32), np.zeros((sizes[1], 5), np.int32), np.zeros(sizes[2], np.int32)
    assert fn(*args, blocks.ctypes.data, segs.ctypes.data, place.ctypes.data) == 0
    nweight, blk = int(sizes[3]), int(sizes[4])
    t = adj_tables(lib, N, order, e, prec)
    assert blk == (4 if prec == "fp64" else 8) and len(place) == len(t["ent"]) and np.unique(place).size == place.size
    rng = np.random.default_rng(nshell)
    D, w = rng.standard_normal(nshell), rng.standard_normal(len(place))
    weight = np.zeros(nweight)
    weight[place] = w
    G = np.zeros(nshell + blk)
    # no warp gives up while another works on its unit: its multiply-adds alone, all 16 warps at work, four times
    unit = int(blocks[:, 4].max()) * 16 * (2 * blk * 16 if prec == "fp64" else 2 * blk * 8 // 4)
    assert sizes[5] >= 4_000_000_000 + 4 * unit
    assert sorted(blocks[:, 0].tolist()) == list(range(0, nshell, blk)) and np.all(np.diff(blocks[:, 4]) <= 0)  # heavy first
    ranges = sorted((b[3], b[3] + b[4]) for b in blocks.tolist())
    assert all(a[1] <= b[0] and b[0] % 8 == 0 for a, b in zip(ranges, ranges[1:]))  # whole batches of 8 records each
    assert ((ranges[-1][1] + 7) // 8) * 8 * 2 * blk <= nweight
    for m0, seg0, nseg, rec0, nrec in blocks.tolist():
        rec = rec0
        for a, j0, j1, i0, count in segs[seg0:seg0 + nseg].tolist():
            assert count > 0 and 0 <= i0 and i0 + count <= nshell and 0 <= j0 <= j1 < nshell and (order < 4 or 0 <= a < nshell)
            for r in range(count):
                for h, j in enumerate((j0, j1)[:2 if order >= 3 else 1]):
                    p = D[i0 + r] * (D[j] if order >= 3 else 1.0) * (D[a] if order == 4 else 1.0)
                    G[m0:m0 + blk] += weight[(rec * 2 + h) * blk:(rec * 2 + h + 1) * blk] * p
                rec += 1
        assert rec - rec0 == nrec
    ref = definition(t, order, nshell, D, w)
    assert np.allclose(G[:nshell], ref, rtol=0, atol=1e-9 * max(1.0, np.abs(ref).max())) and np.all(G[nshell:] == 0)

"""The tensor-core contraction's compact layout of orders 4 and 5 (rows sorted by their last legs, three-leg rows
for n = 5): every bin's slot is the product of exactly its shells, no slot is used twice, and the
plans that the plain layout refuses stay refused.  Host tables only."""
import numpy as np
import pytest

import fieldgen
import oracle
import paper_1904_11055_gb300 as ps
from paper_1904_11055_gb300 import build as psbuild
from test_host_tables_cpu import STATUS, check_pipeline_teams, tc_tables


@pytest.fixture(scope="module")
def lib():
    psbuild.build()
    return ps.load_library()


@pytest.mark.parametrize("N,order,nshell,width,ell", [
    (256, 4, 32, 1.5, 0), (160, 4, 26, 1.5, 0), (128, 4, 17, 1.0, 0), (48, 4, 3, 1.0, 0), (64, 4, 12, 1.0, 2),
    (128, 5, 17, 1.0, 0), (128, 5, 20, 1.0, 0), (256, 5, 20, 2.0, 0), (128, 5, 16, 1.0, 0), (64, 5, 10, 1.0, 0),
    (48, 5, 3, 1.0, 0), (64, 5, 6, 1.0, 2)])
def test_every_bin_has_its_own_slot_of_its_own_product(lib, N, order, nshell, width, ell):
    e = fieldgen.unit_edges(nshell, width)
    rc, t = tc_tables(lib, N, order, e, flags=0, ell=ell)
    assert rc == 0
    bins, bm = oracle.enumerate_bins(e, order), t["binmap"]
    check_pipeline_teams(t)
    group = t["ctas"][bm[:, 0], 0]
    assert np.unique(group * (256 * 128) + bm[:, 2]).size == len(bins)
    shift = nshell if ell else 0
    owner = {}  # (group, accumulator column) -> (M tile, column record)
    for g, (mt_off, nmt, col_off, ncol, acc_cols) in enumerate(t["groups"]):
        assert 1 <= nmt <= 4 and ncol <= 256 and acc_cols <= 256
        for m in range(mt_off, mt_off + nmt):
            _, run_off, nrun = t["mtiles"][m]
            for n0, nn, acc, _ in t["runs"][run_off:run_off + nrun]:
                for j in range(nn):
                    assert (g, acc + j) not in owner
                    owner[g, acc + j] = (m, col_off + n0 + j)
    for b, legs in enumerate(bins.astype(int) - 1):
        m, col = owner[int(group[b]), int(bm[b, 2]) // 128]
        row = t["rowf"][t["mtiles"][m, 0] + int(bm[b, 2]) % 128]
        want = [int(v) for v in legs]
        want[0] += shift
        assert [int(v) for v in row if v >= 0] + [int(v) for v in t["colf"][col] if v >= 0] == want


@pytest.mark.parametrize("order,nshell,ell", [(4, 35, 0), (4, 64, 0), (4, 20, 2), (5, 17, 2), (5, 20, 2)])
def test_refused_plans_stay_refused(lib, order, nshell, ell):
    rc, _ = tc_tables(lib, 256, order, fieldgen.unit_edges(nshell), flags=ps.POLY_ALLOW_ALIAS, ell=ell)
    assert rc == STATUS["POLY_ERR_UNSUPPORTED"]


@pytest.mark.parametrize("nshell,groups,teams", [(26, 2, 3), (27, 4, 3), (28, 4, 2), (32, 4, 3), (33, 7, 3), (34, 6, 2)])
def test_order_4_takes_the_faster_layout_and_the_teams_that_fit(lib, nshell, groups, teams):
    """The measured choice at 256^3 in shells of 1.5: 27 and 33 shells keep the plain layout's groups and three teams (fewer
    groups of two teams take longer), 32 take the compact one's with three."""
    rc, t = tc_tables(lib, 256, 4, fieldgen.unit_edges(nshell, 1.5))
    assert rc == 0
    check_pipeline_teams(t)
    assert (len(t["groups"]), t["teams"]) == (groups, teams)

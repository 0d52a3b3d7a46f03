"""The graph builder takes four consecutive particles per warp: systems whose
size is no multiple of it, groups that span cells, rows and members, and dense
cells (more than 32 candidates per run, jittered block at a larger h) give
exactly the FP64 reference's ordered pairs, each row ascending."""
import numpy as np
import pytest

import __graft_entry__  # noqa: F401
from oracle import sur_oracle as so
from paper_1210_1017_gb300 import cases
from paper_1210_1017_gb300 import sph as S
from paper_1210_1017_gb300 import surrogate as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    return t


@pytest.mark.parametrize("n,copies,h_over_dp,radius", [
    (3, 1, 1.3, 1.0), (6, 3, 1.3, 1.0), (33, 1, 1.3, 0.8), (413, 2, 1.3, 1.0),
    (1201, 1, 2.2, 1.0), (1202, 1, 0.8, 0.6), (1203, 3, 1.3, 0.7)])
def test_graph_equals_the_reference_pairs(torch, n, copies, h_over_dp, radius):
    case = cases.random_block(n, seed=n, jitter=0.3, h_over_dp=h_over_dp)
    sim = S.Simulation.from_ensemble(cases.ensemble([case] * copies))
    sim.build_cells()
    sur = U.Surrogate(sim, layers=1, train=False, v_scale=0.5, radius=radius,
                      max_edges=case.n * copies * 400)
    sur.set_params(so.init_params(1, seed=1))
    N = case.n * copies
    sur.forward(torch.zeros((N, 15), device="cuda"), torch.zeros((N, 3), device="cuda"))
    sim.synchronize()
    rowptr, col = sur.read_graph()
    rowptr, col = rowptr.astype(np.int64), col.astype(np.int64)
    src = np.repeat(np.arange(N), np.diff(rowptr))
    inner = np.ones(len(col), bool)
    inner[rowptr[:-1][np.diff(rowptr) > 0]] = False
    assert np.all(np.diff(col, prepend=-1)[inner] > 0)
    ids = sim.download()["ids"].astype(np.int64)
    g_src, g_dst = ids[src], ids[col]
    order = np.lexsort((g_dst, g_src))
    pos = case.pos[np.argsort(case.ids)]
    rs, rd = so.graph(pos, radius * case.h)
    ref_src = np.concatenate([rs + q * case.n for q in range(copies)])
    ref_dst = np.concatenate([rd + q * case.n for q in range(copies)])
    assert np.array_equal(g_src[order], ref_src)
    assert np.array_equal(g_dst[order], ref_dst)
    sim.close()

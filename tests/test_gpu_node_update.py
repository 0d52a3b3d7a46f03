"""The fused node update (both layers of the node network and the next layer's
node terms, per 128-node tile) at node counts that cut the tiles elsewhere: one
tile, ragged last tiles, several tiles per block.  Every value of a node depends
on its own rows only, so each of several copies of a block gives exactly the
accelerations of one block; one block is compared with the FP64 reference in
test_gpu_surrogate_net.py."""
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


def _acc(torch, case, copies, layers, w):
    sim = S.Simulation.from_ensemble(cases.ensemble([case] * copies))
    sim.build_cells()
    hist = np.random.default_rng(3).normal(0, 0.4, (case.n, 15)).astype(np.float32)
    hist[:case.n_bound] = 0
    sur = U.Surrogate(sim, layers=layers, train=False, v_scale=0.5)
    sur.set_params(w)
    acc = torch.zeros((case.n * copies, 3), dtype=torch.float32, device="cuda")
    sur.forward(torch.tensor(np.tile(hist, (copies, 1)), device="cuda"), acc)
    sim.synchronize()
    out = acc.cpu().numpy().reshape(copies, case.n, 3)
    sim.close()
    return out


@pytest.mark.parametrize("n,copies,layers", [(3, 1, 1), (3, 43, 2), (127, 3, 3), (130, 2, 2),
                                             (1000, 45, 2)])
def test_copies_of_a_block_move_alike(torch, n, copies, layers):
    case = cases.random_block(n, seed=n, jitter=0.3)
    w = so.init_params(layers, seed=n + 2)
    one = _acc(torch, case, 1, layers, w)[0]
    many = _acc(torch, case, copies, layers, w)
    assert np.isfinite(one).all() and np.abs(one).max() > 0
    for q in range(copies):
        assert np.array_equal(many[q], one), q

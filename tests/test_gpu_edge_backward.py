"""The fused backward pass of the edge update at edge counts that cut its
128-edge tiles at other places: the gradients of 2^k copies of a particle block
are those of one block (the loss is a mean, and 1 / n_fluid scales by a power
of two without rounding), so every per-edge value is the same bit for bit and
only the order of the FP32 sums over edges and nodes differs.  Against the FP64
reference, one block is compared in test_gpu_surrogate_net.py.

Bar: a sum of E terms in FP32 in another order is off by about 2^-24 sqrt(log E)
of its partial sums, some 1e-6 of the result for terms of random sign; 1e-4 of
a layer's gradient norm leaves room for cancellation in the bias gradients."""
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


def _grads(torch, case, copies, layers, w):
    sim = S.Simulation.from_ensemble(cases.ensemble([case] * copies))
    sim.build_cells()
    rng = np.random.default_rng(5)
    hist = rng.normal(0, 0.4, (case.n, 15)).astype(np.float32)
    hist[:case.n_bound] = 0
    target = rng.normal(0, 1.0, (case.n, 3)).astype(np.float32)
    d_hist = torch.tensor(np.tile(hist, (copies, 1)), device="cuda")
    d_target = torch.tensor(np.tile(target, (copies, 1)), device="cuda")
    sur = U.Surrogate(sim, layers=layers, train=True, v_scale=0.5)
    sur.set_params(w)
    acc = torch.zeros((case.n * copies, 3), dtype=torch.float32, device="cuda")
    sur.forward(d_hist, acc)
    sur.backward(d_target)
    g = sur.grads().astype(np.float64)
    edges = sur.num_edges
    # a second pass gives the same bits
    sur.forward(d_hist, acc)
    sur.backward(d_target)
    assert np.array_equal(g, sur.grads().astype(np.float64))
    sim.close()
    return g, edges


@pytest.mark.parametrize("n,copies", [(5, 2), (5, 8), (60, 4), (300, 32), (1100, 16)])
def test_gradients_of_copies_equal_those_of_one_block(torch, n, copies):
    layers = 2
    case = cases.random_block(n, seed=n, jitter=0.3)
    w = so.init_params(layers, seed=n + 1)
    g1, e1 = _grads(torch, case, 1, layers, w)
    gk, ek = _grads(torch, case, copies, layers, w)
    assert ek == copies * e1
    o = 0
    for name, ki, ko, has_b in so.layer_shapes(layers):
        for part, size in (("W", ki * ko), ("b", ko if has_b else 0)):
            a, b = gk[o:o + size], g1[o:o + size]
            o += size
            norm = np.linalg.norm(b)
            assert np.linalg.norm(a - b) <= 1e-4 * norm + 1e-12, (name, part, norm)
    assert o == len(g1)

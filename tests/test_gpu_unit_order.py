"""Interaction blocks that take dense units (candidates read from global memory,
their lists in the staging area) and staged ones in turn: what one unit leaves in
shared and tensor memory must not reach the next one's staging copies and
products.  A sparse gas (more units than any shape has blocks) with clumps of
2,000 particles in single cells; rates equal from launch to launch bit for bit,
and within the 2e-5 bar of the FP64 oracle (accelerations relative to the sum of
the pair terms)."""
import numpy as np
import pytest

import __graft_entry__
import oracle
from paper_1210_1017_gb300 import cases
from paper_1210_1017_gb300 import sph as S

pytestmark = pytest.mark.gpu
H, SIDE, CLUMP = 0.05, 3.0, 2000


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    yield


def _clumped_gas():
    rng = np.random.default_rng(12)
    c = cases.random_block(6000 + 6 * CLUMP, seed=12, bound_layers=0)
    m = c.pos.shape[0]
    c.pos = rng.uniform(0, SIDE, (m, 3))
    for k in range(6):
        sel = slice(k * CLUMP, (k + 1) * CLUMP)
        c.pos[sel] = rng.uniform(0.3, SIDE - 0.3, 3) + rng.uniform(-0.04, 0.04, (CLUMP, 3))
    c.vel = rng.uniform(-1, 1, (m, 3)).astype(np.float32)
    c.h, c.n_bound = H, m // 5
    c.ids = rng.permutation(m).astype(np.uint32)
    c.dmin, c.dmax = cases.domain_for(c.pos, H, SIDE, 4 * H)
    return c


def test_dense_and_staged_units_in_turn():
    case = _clumped_gas()
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    st = sim.download()
    ref = oracle.Oracle(case.params()).interact(
        oracle.State(st["pos"], st["vel"], st["rho"], st["ids"]))
    fluid = st["ids"] >= case.n_bound
    off = sim.read(S.SPH_ARRAY_CELL_OFF)
    assert np.diff(off[:-1].astype(np.int64)).max() >= 200
    for v in range(S.sph_num_variants()):
        sim.set_variant(v)
        assert sim.units().shape[0] > 608          # four blocks on each of 152 SMs
        first = None
        for _ in range(4):
            sim.interact()
            sim.check()
            ace = sim.read(S.SPH_ARRAY_ACE)
            first = ace if first is None else first
            assert np.array_equal(ace, first), v
        ea = np.linalg.norm(first[fluid, :3] - ref["a"][fluid], axis=1) / \
            np.maximum(ref["sa"][fluid], 1e-300)
        assert ea.max() <= 2e-5, (v, ea.max())
    sim.close()


@pytest.mark.parametrize("h_over_dp", [1.1, 1.7])
def test_units_of_one_and_of_several_pieces(h_over_dp):
    """Units of at most 256 candidates (one product) and of several: the next
    unit's product overwrites accumulators that the last piece's readers hold."""
    case = cases.random_block(30000, seed=13, h_over_dp=h_over_dp, jitter=0.2)
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    st = sim.download()
    ref = oracle.Oracle(case.params()).interact(
        oracle.State(st["pos"], st["vel"], st["rho"], st["ids"]))
    fluid = st["ids"] >= case.n_bound
    for v in range(7):
        sim.set_variant(v)
        first = None
        for _ in range(4):
            sim.interact()
            sim.check()
            ace = sim.read(S.SPH_ARRAY_ACE)
            first = ace if first is None else first
            assert np.array_equal(ace, first), v
        ea = np.linalg.norm(first[fluid, :3] - ref["a"][fluid], axis=1) / ref["sa"][fluid]
        assert ea.max() <= 2e-5, (v, ea.max())
    sim.close()

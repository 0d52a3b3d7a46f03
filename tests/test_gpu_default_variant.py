"""A context that has not been tuned takes an interaction shape that stages its
units at its particles per cell: the rates of a fresh context equal, bit for bit,
those of the shape that the rule names, on both sides of the line."""
import numpy as np
import pytest

import __graft_entry__
from paper_1210_1017_gb300 import cases
from paper_1210_1017_gb300 import sph as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    yield


@pytest.mark.parametrize("h_over_dp,variant", [(1.3, 0), (1.6, 0), (1.61, 13), (2.1, 13), (3.0, 13)])
def test_shape_of_a_fresh_context(h_over_dp, variant):
    case = cases.random_block(4000, seed=41, h_over_dp=h_over_dp, jitter=0.2)
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    sim.interact()
    fresh = sim.read(S.SPH_ARRAY_ACE)
    others = []
    for v in (0, 13):
        sim.set_variant(v)
        sim.interact()
        others.append(sim.read(S.SPH_ARRAY_ACE))
    sim.check()
    assert not np.array_equal(*others)           # the two shapes round differently
    assert np.array_equal(fresh, others[(0, 13).index(variant)])
    sim.close()

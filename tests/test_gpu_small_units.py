"""The interaction in small units of length (h = 0.1 um in metres): the kernel
gradient's factor, about 2 / h^5, is near the top of the FP32 range, and the pads
of idle lanes, 32 cells away, must not overflow it.  Every variant finite and
within the 2e-5 bar of the FP64 oracle, both kernels."""
import dataclasses

import numpy as np
import pytest

import __graft_entry__
import oracle
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


@pytest.mark.parametrize("kernel", ["wendland", "cubic"])
def test_tenth_of_a_micrometre(kernel):
    case = cases.random_block(4000, seed=9, jitter=0.3)
    f = 1e-7 / case.h
    case = dataclasses.replace(case, pos=case.pos * f, dp=case.dp * f, h=case.h * f, kernel=kernel)
    case.dmin, case.dmax = cases.domain_for(case.pos, case.h, float(case.pos[:, 2].max()), 4 * case.h)
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    st = sim.download()
    ref = oracle.Oracle(case.params()).interact(
        oracle.State(st["pos"], st["vel"], st["rho"], st["ids"]))
    fluid = st["ids"] >= case.n_bound
    for v in range(S.sph_num_variants()):
        sim.set_variant(v)
        sim.interact()
        sim.check()
        ace = sim.read(S.SPH_ARRAY_ACE)
        ea = np.linalg.norm(ace[fluid, :3] - ref["a"][fluid], axis=1) / ref["sa"][fluid]
        assert ea.max() <= 2e-5, (v, ea.max())
    sim.close()

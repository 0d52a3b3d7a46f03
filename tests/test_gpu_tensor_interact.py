"""The tensor-core shapes of the interaction (variants 0-6) where they can go
wrong: units across empty cells and at the span limit, cells dense enough to
fill the lists of hit words (several pair phases per unit) and to overflow the
staging (global-memory path), units of one to a few particles, several
instances.  Rates within the 2e-5 bar of the FP64 oracle (accelerations
relative to the sum of the pair terms, density rates to the sum of m F0
(1 - q/2)^2 |v_ij| |r_ij|, which bounds the rounding of the dot products and of
F = F0 (1 - q/2)^3: a lone neighbour's v.r may cancel, and its q be near 2);
an earlier shape (variant 13) under the same bars; FP32 neighbour counts equal to the FP64 ones but
for pairs within 1e-6 of the support."""
import numpy as np
import pytest

import __graft_entry__
import oracle
from paper_1210_1017_gb300 import cases
from paper_1210_1017_gb300 import sph as S

pytestmark = pytest.mark.gpu
TENSOR_VARIANTS = range(7)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    yield


def _gas(n, box, h, seed):
    """Particles at random in a box (sparse: most cells empty)."""
    rng = np.random.default_rng(seed)
    c = cases.random_block(n, seed=seed, bound_layers=0)
    m = c.pos.shape[0]
    c.pos = rng.uniform(0, 1, (m, 3)) * np.array(box)
    c.vel = rng.uniform(-1, 1, (m, 3)).astype(np.float32)
    c.h, c.n_bound = h, m // 5
    c.ids = rng.permutation(m).astype(np.uint32)
    c.dmin, c.dmax = cases.domain_for(c.pos, h, float(c.pos[:, 2].max()), 4 * h)
    return c


CASES = {
    # about one particle in three cells: units span gaps and many cells
    "sparse_rows": lambda: _gas(3000, (40.0, 1.0, 1.0), 0.05, 1),
    "sparse_box": lambda: _gas(2000, (3.0, 2.0, 2.0), 0.05, 2),
    # about 2, 10 and 60 particles per cell
    "two_per_cell": lambda: _gas(4000, (1.6, 0.8, 0.8), 0.04, 3),
    "ten_per_cell": lambda: _gas(6000, (1.6, 0.5, 0.5), 0.04, 4),
    "dense_2dp": lambda: cases.random_block(4000, seed=5, h_over_dp=2.0, jitter=0.2),
    "dense_3dp": lambda: cases.random_block(3000, seed=6, h_over_dp=3.0, jitter=0.2),
    "one_and_two": lambda: _gas(2, (0.05, 0.05, 0.05), 0.05, 7),
    "moving_dam": lambda: cases.c1_dam_break(shuffle_seed=4),
}


@pytest.mark.parametrize("name", list(CASES))
def test_rates_and_counts(name):
    case = CASES[name]()
    sim = S.Simulation.from_case(case)
    if name == "moving_dam":
        sim.step(60)
    sim.build_cells()
    st = sim.download()
    ref = oracle.Oracle(case.params()).interact(
        oracle.State(st["pos"], st["vel"], st["rho"], st["ids"]))
    fluid = st["ids"] >= case.n_bound
    c64 = sim.neighbour_counts_fp64().astype(np.int64)
    # per particle: pairs within 1e-6 of the support, and the density scale
    near, sd = np.zeros(case.n, np.int64), np.zeros(case.n)
    r2 = (2 * case.h) ** 2
    for k in range(0, case.n, 500):
        d2 = ((st["pos"][k:k + 500, None] - st["pos"][None]) ** 2).sum(-1)
        near[k:k + 500] = (np.abs(d2 - r2) < 1e-6 * r2).sum(1)
        v2 = ((st["vel"][k:k + 500, None] - st["vel"][None]).astype(np.float64) ** 2).sum(-1)
        F = 5 * 21 / (16 * np.pi * case.h ** 5) * np.maximum(1 - np.sqrt(d2 / r2), 0) ** 2
        sd[k:k + 500] = case.mass * (F * np.sqrt(v2 * d2)).sum(1)
    for v in [*TENSOR_VARIANTS, 13]:
        sim.set_variant(v)
        sim.interact(counts=True)
        sim.check()
        ace = sim.read(S.SPH_ARRAY_ACE)
        ea = np.linalg.norm(ace[fluid, :3] - ref["a"][fluid], axis=1) / \
            np.maximum(ref["sa"][fluid], 1e-300)
        ed = np.abs(ace[:, 3] - ref["drho"]) / np.where(sd > 0, sd, 1.0)
        assert ea.max() <= 2e-5 and ed.max() <= 2e-5, (name, v, ea.max(), ed.max())
        nnb = sim.read(S.SPH_ARRAY_NNB).astype(np.int64)
        assert np.all(np.abs(nnb - c64) <= near), (name, v)
    sim.close()


def test_members_of_an_ensemble_equal_their_single_runs():
    members = [cases.ensemble_instance(s) for s in cases.ensemble_specs(3, seed=11)]
    ens = cases.ensemble(members)
    sim = S.Simulation.from_ensemble(ens)
    alone = [S.Simulation.from_case(m) for m in members]
    for v in (0, 1):
        sim.set_variant(v)
        sim.build_cells()
        sim.interact()
        ace, ids = sim.read(S.SPH_ARRAY_ACE), sim.download()["ids"]
        for k, one in enumerate(alone):
            one.set_variant(v)
            one.build_cells()
            one.interact()
            sel = (ids >= ens.id_base[k]) & (ids < ens.id_base[k + 1])
            assert np.array_equal(ace[sel], one.read(S.SPH_ARRAY_ACE)), (v, k)
    for s in alone + [sim]:
        s.close()

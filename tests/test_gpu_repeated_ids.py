"""The sub-domain selection where an id occurs twice: once in each of the two
labels, twice in one label, and with a particle of neither.  Every labelled
particle comes out once, under its label, in ascending id (equal ids of one label
in any order), with its own position, velocity and density."""
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


@pytest.mark.parametrize("pairs", ["across", "within", "outside", "all"])
def test_every_selected_particle_comes_out_once(pairs):
    case = cases.random_block(9000, seed=23, jitter=0.4)
    case.n_bound = 0
    x = case.pos[:, 0]
    lo, hi = float(np.quantile(x, 0.3)), float(np.quantile(x, 0.6))
    lab = np.where(x < lo, 1, np.where(x >= hi, 2, 0))
    one, two, none = (np.nonzero(lab == k)[0] for k in (1, 2, 0))
    if pairs in ("across", "all"):
        case.ids[two[:40]] = case.ids[one[:40]]
    if pairs in ("within", "all"):
        case.ids[one[50:60]] = case.ids[one[60:70]]
    if pairs in ("outside", "all"):
        case.ids[none[:20]] = case.ids[one[80:100]]
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    for _ in range(3):
        got = sim.subdomain_select(S.SPH_SUBDOMAIN_MIGRATE, lo, hi)
        assert got["counts"].tolist() == [none.size, one.size, two.size]
        at = 0
        for sel in (one, two):
            part = slice(at, at + sel.size)
            at += sel.size
            assert np.array_equal(got["ids"][part], np.sort(case.ids[sel]))
            rows = [np.column_stack([i, p, v, r]) for i, p, v, r in (
                (got["ids"][part], got["pos"][part], got["vel"][part], got["rho"][part]),
                (case.ids[sel], case.pos[sel], case.vel[sel].astype(np.float32),
                 case.rho[sel].astype(np.float32)))]
            a, b = (r[np.lexsort(r.T[::-1])] for r in rows)
            assert np.array_equal(a, b)
    sim.check()
    sim.close()


@pytest.mark.parametrize("n", [40, 1200, 4000])
def test_few_ids_above_n_are_sorted_in_place(n):
    """A selection of at most one tile of pairs, by the sort (ids up to 2^32 - 1)."""
    case = cases.random_block(n, seed=24, jitter=0.4)
    case.n_bound = 0
    case.ids = (np.uint32(0xffffffff) - np.random.default_rng(1).permutation(
        4 * case.n)[:case.n].astype(np.uint32) * np.uint32(1001))
    x = case.pos[:, 0]
    lo, hi = float(np.quantile(x, 0.4)), float(np.quantile(x, 0.6))
    lab = np.where(x < lo, 1, np.where(x >= hi, 2, 0))
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    got = sim.subdomain_select(S.SPH_SUBDOMAIN_MIGRATE, lo, hi)
    sel = np.nonzero(lab)[0]
    sel = sel[np.lexsort((case.ids[sel], lab[sel]))]
    assert np.array_equal(got["ids"], case.ids[sel])
    for key in ("pos", "vel", "rho"):
        assert np.array_equal(got[key], getattr(case, key)[sel]), key
    sim.close()


def test_calls_in_turn_leave_nothing_behind():
    """Empty, full, refused and repeated-id selections in turn on one context: each
    as on a context of its own (the bit maps are cleared by the call that used them)."""
    case = cases.random_block(5000, seed=25, jitter=0.4)
    case.n_bound = 0
    x = case.pos[:, 0]
    lo, hi = float(np.quantile(x, 0.3)), float(np.quantile(x, 0.6))
    one = np.nonzero(x < lo)[0]
    ids = case.ids.copy()
    twice = case.ids.copy()
    twice[one[:3]] = twice[one[3:6]]
    wide = (float(x.min()) - 1.0, float(x.max()) + 1.0)
    sim = S.Simulation(case.params(), case.n)

    def call(of, bounds):
        alone = S.Simulation(case.params(), case.n)
        got = []
        for s in (sim, alone):
            s.upload(case.pos, case.vel, case.rho, of)
            s.build_cells()
            got.append(s.subdomain_select(S.SPH_SUBDOMAIN_MIGRATE, *bounds))
        alone.close()
        assert got[0]["counts"].tolist() == got[1]["counts"].tolist()
        assert np.array_equal(got[0]["ids"], got[1]["ids"])
        if of is ids:
            for key in ("pos", "vel", "rho"):
                assert np.array_equal(got[0][key], got[1][key]), key
        return got[0]["ids"].size

    small = np.empty(1, np.uint32)
    for of, bounds in ((ids, wide), (ids, (lo, hi)), (ids, wide), (twice, (lo, hi)), (ids, (hi, hi + 1.0)),
                       (ids, (lo, hi)), (twice, wide), (ids, (lo, hi))):
        m = call(of, bounds)
        assert (m == 0) == (bounds is wide)
        if m:
            with pytest.raises(S.SphError, match="SPH_ERR_CAPACITY"):
                S.sph_subdomain_select(sim.ctx, S.SPH_SUBDOMAIN_MIGRATE, *bounds, 1, None, None, None, small)
    sim.close()

"""A member that has ended keeps its state whatever rates the context's last run
left behind: a run that went non-finite, then a sound state uploaded into the
same context with the first member past its end time."""
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


def test_an_ended_member_after_a_run_that_went_non_finite():
    members = [cases.ensemble_instance(s) for s in cases.ensemble_specs(2, seed=5)]
    ens = cases.ensemble(members, t_end=3e-3)
    sim = S.Simulation.from_ensemble(ens)
    bad = np.ascontiguousarray(ens.vel, np.float32).copy()
    bad[np.arange(ens.n) % 7 == 0] = np.nan
    sim.upload(ens.pos, bad, ens.rho, ens.ids)
    sim.build_cells()
    sim.interact()
    with pytest.raises(S.SphError, match="SPH_ERR_NONFINITE"):
        sim.check()
    S.sph_clear_status(sim.ctx)
    assert np.isnan(sim.read(S.SPH_ARRAY_ACE)).any(axis=1).sum() > ens.n // 4
    sim.upload(ens.pos, ens.vel, ens.rho, ens.ids)
    sim.set_instance_state(np.array([1.0, 0.0]))
    sim.step(3)
    sim.check()
    st = sim.download()
    back = np.argsort(st["ids"])
    one, two = ens.member_slice(0), ens.member_slice(1)
    for key in ("pos", "vel", "rho"):
        assert np.array_equal(st[key][back][one], getattr(ens, key)[one]), key
        assert np.isfinite(st[key]).all(), key
    assert not np.array_equal(st["vel"][back][two], ens.vel[two])
    sim.close()

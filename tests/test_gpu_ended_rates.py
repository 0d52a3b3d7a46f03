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


def test_a_predictor_step_before_any_evaluation_takes_no_rates():
    """In a workspace of NaNs, dt = 0 as no evaluation has set it."""
    import torch
    case = cases.random_block(500, seed=6, jitter=0.2)
    P = S.make_params(case.params(), 0.0)
    nbytes = int(S.sph_query_sizes(P, case.n).workspace_bytes)
    ws = torch.full((nbytes,), 255, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = S.sph_init(P, case.n, ws.data_ptr(), nbytes, stream.cuda_stream)
    try:
        S.sph_upload(ctx, np.ascontiguousarray(case.pos), np.ascontiguousarray(case.vel, np.float32),
                     np.ascontiguousarray(case.rho, np.float32), np.ascontiguousarray(case.ids))
        S.sph_build_cells(ctx)
        S.sph_predict(ctx)
        n = case.n
        pos, vel = np.empty((n, 3)), np.empty((n, 3), np.float32)
        rho, ids = np.empty(n, np.float32), np.empty(n, np.uint32)
        S.sph_download(ctx, pos, vel, rho, ids)
    finally:
        stream.synchronize()
        S.sph_destroy(ctx)
    back = np.argsort(ids)
    order = np.argsort(case.ids)
    for got, want in ((pos, case.pos), (vel, case.vel), (rho, case.rho)):
        assert np.array_equal(got[back], want[order])

"""A member that has reached its end time before the context's first
evaluation (an ensemble resumed from a checkpoint) keeps its state, whatever
the workspace memory held: its rates are never evaluated, and dt = 0 times
what they hold has to be 0 (not NaN)."""
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


def test_an_ended_member_keeps_its_state_in_a_workspace_of_nans():
    import torch
    members = [cases.ensemble_instance(s) for s in cases.ensemble_specs(2, seed=5)]
    ens = cases.ensemble(members, t_end=3e-3)
    sim = S.Simulation.from_ensemble(ens)
    nbytes = int(sim.sizes.workspace_bytes)
    sim.close()
    # all bits set (a NaN in every format) under the library's feet
    ws = torch.full((nbytes,), 255, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = S.sph_init_batch(sim.P, sim.members, ws.data_ptr(), nbytes, stream.cuda_stream)
    try:
        S.sph_upload(ctx, np.ascontiguousarray(ens.pos), np.ascontiguousarray(ens.vel, np.float32),
                     np.ascontiguousarray(ens.rho, np.float32), np.ascontiguousarray(ens.ids))
        S.sph_set_instance_state(ctx, np.array([1.0, 0.0]))      # the first member has ended
        S.sph_step(ctx, 3)
        S.sph_check(ctx)
        n = ens.n
        pos, vel = np.empty((n, 3)), np.empty((n, 3), np.float32)
        rho, ids = np.empty(n, np.float32), np.empty(n, np.uint32)
        S.sph_download(ctx, pos, vel, rho, ids)
    finally:
        stream.synchronize()
        S.sph_destroy(ctx)
    back = np.argsort(ids)
    one = ens.member_slice(0)
    assert np.array_equal(pos[back][one], ens.pos[one])
    assert np.array_equal(vel[back][one], ens.vel[one]) and np.array_equal(rho[back][one], ens.rho[one])
    assert np.isfinite(pos).all() and np.isfinite(vel).all() and np.isfinite(rho).all()
    two = ens.member_slice(1)
    assert not np.array_equal(vel[back][two], ens.vel[two])

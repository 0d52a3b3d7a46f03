"""Device arrays at addresses that only a copy can take (positions behind an odd
number of 4-byte words, everything at odd bytes): upload, download, download by id
and the sub-domain selection give what they give with aligned arrays."""
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


class _At:
    """An address in device memory (``off`` bytes into a byte tensor)."""

    def __init__(self, nbytes, off, data=None):
        import torch
        self.buf = torch.full((nbytes + 64,), 255, dtype=torch.uint8, device="cuda")
        self.off, self.nbytes = off, nbytes
        if data is not None:
            raw = torch.from_numpy(np.frombuffer(data.tobytes(), np.uint8).copy())
            self.buf[off:off + nbytes] = raw.cuda()

    def data_ptr(self):
        return self.buf.data_ptr() + self.off

    def numpy(self, dtype, shape):
        raw = self.buf[self.off:self.off + self.nbytes].cpu().numpy()
        return np.frombuffer(raw.tobytes(), dtype).reshape(shape)


@pytest.mark.parametrize("off", [4, 1, 2, 8])
def test_transfers_and_selection(off):
    import torch
    case = cases.random_block(3001, seed=31, jitter=0.3)
    n = case.n
    ref = S.Simulation.from_case(case)
    sim = S.Simulation(case.params(), n)
    up = [_At(a.nbytes, off, a) for a in (np.ascontiguousarray(case.pos),
                                          np.ascontiguousarray(case.vel, np.float32),
                                          np.ascontiguousarray(case.rho, np.float32),
                                          np.ascontiguousarray(case.ids, np.uint32))]
    torch.cuda.synchronize()
    S.sph_upload(sim.ctx, *up)
    sizes = [24 * n, 12 * n, 4 * n, 4 * n]
    shapes = [(np.float64, (n, 3)), (np.float32, (n, 3)), (np.float32, (n,)), (np.uint32, (n,))]
    for s in (ref, sim):
        s.step(3)
        s.build_cells()
        s.check()
    want = ref.download()
    out = [_At(b, off) for b in sizes]
    torch.cuda.synchronize()
    S.sph_download(sim.ctx, *out)
    for key, o, (dt, sh) in zip(("pos", "vel", "rho", "ids"), out, shapes):
        assert np.array_equal(o.numpy(dt, sh), want[key]), key
    by_id = [np.empty((n, 3)), np.empty((n, 3), np.float32), np.empty(n, np.float32)]
    S.sph_download_by_id(ref.ctx, *by_id)
    out = [_At(b, off) for b in sizes[:3]]
    torch.cuda.synchronize()
    S.sph_download_by_id(sim.ctx, *out)
    for w, o, (dt, sh) in zip(by_id, out, shapes):
        assert np.array_equal(o.numpy(dt, sh), w)
    x = want["pos"][:, 0]
    lo, hi = float(np.quantile(x, 0.3)), float(np.quantile(x, 0.6))
    sel = ref.subdomain_select(S.SPH_SUBDOMAIN_MIGRATE, lo, hi)
    m = sel["ids"].size
    assert m > 500
    out = [_At(b * m // n, off) for b in sizes]
    torch.cuda.synchronize()
    S.sph_subdomain_select(sim.ctx, S.SPH_SUBDOMAIN_MIGRATE, lo, hi, m, *out)
    for key, o, (dt, sh) in zip(("pos", "vel", "rho", "ids"), out, shapes):
        assert np.array_equal(o.numpy(dt, (m,) + sh[1:]), sel[key]), key
    ref.close()
    sim.close()

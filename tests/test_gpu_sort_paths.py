"""The radix sort at the sizes where its path changes (one tile of 4,096 pairs
in one block; up to 96 tiles without the scan of the tile counts; more) and on
key arrays that are not 16-byte aligned, against numpy's stable sort; the
sub-domain selection by bit maps of the ids against the sorted path (ids that
repeat, ids at and above n) and into device arrays.  Everything exact."""
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


TILE = 4096


@pytest.mark.parametrize("bits", [1, 8, 13, 32])
@pytest.mark.parametrize("n", [1, 33, 257, TILE - 1, TILE, TILE + 1, 96 * TILE, 96 * TILE + 1,
                               97 * TILE + 7, 1000003])
def test_sizes_and_key_bits(n, bits):
    import torch
    rng = np.random.default_rng(n + bits)
    keys = rng.integers(0, 1 << bits, n, dtype=np.uint64).astype(np.uint32)
    vals = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    order = np.argsort(keys, kind="stable")
    for off in (0, 1):                       # off 1: not 16-byte aligned
        pad = np.zeros(off, np.uint32)
        k = torch.from_numpy(np.concatenate([pad, keys]).view(np.int32)).cuda()[off:]
        v = torch.from_numpy(np.concatenate([pad, vals]).view(np.int32)).cuda()[off:]
        ko, vo = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(
            n, dtype=torch.int32, device="cuda")
        nb = int(S.lib().sph_radix_sort_scratch_bytes(n))
        scratch = torch.randint(0, 255, (nb,), dtype=torch.uint8, device="cuda")   # stale contents
        st = torch.cuda.current_stream().cuda_stream
        for values in (v, None):
            S.sph_radix_sort_pairs(k, values, ko, vo, n, bits, scratch, nb, st)
            S.sph_radix_sort_status(scratch, nb, n, st)
            assert np.array_equal(ko.cpu().numpy().view(np.uint32), keys[order])
            want = vals[order] if values is not None else order.astype(np.uint32)
            assert np.array_equal(vo.cpu().numpy().view(np.uint32), want)



@pytest.mark.parametrize("ids", ["dense", "repeated", "above_n"])
def test_selection_is_in_label_id_order(ids):
    case = cases.random_block(9000, seed=21, jitter=0.4)
    n = case.n
    if ids == "repeated":                    # one id twice: below n, not distinct
        case.ids[case.ids == 17] = 18
    if ids == "above_n":
        case.ids[case.ids == 17] = n
    case.n_bound = 0
    sim = S.Simulation.from_case(case)
    sim.build_cells()
    st = sim.download()
    x = st["pos"][:, 0]
    for mode, xlo, xhi in ((S.SPH_SUBDOMAIN_MIGRATE, np.quantile(x, 0.3), np.quantile(x, 0.6)),
                           (S.SPH_SUBDOMAIN_EDGE, x.min(), x.max())):
        w = 2 * case.h
        lab = np.where(x < xlo, 1, np.where(x >= xhi, 2, 0)) if mode == S.SPH_SUBDOMAIN_MIGRATE \
            else np.where((x >= xlo) & (x < xlo + w), 1, np.where((x >= xhi - w) & (x < xhi), 2, 0))
        got = sim.subdomain_select(mode, float(xlo), float(xhi))
        sel = np.nonzero(lab)[0]
        sel = sel[np.lexsort((st["ids"][sel], lab[sel]))]
        assert sel.size > 500
        assert got["counts"].tolist() == [int((lab == k).sum()) for k in range(3)]
        assert np.array_equal(got["ids"], st["ids"][sel])
        if ids != "repeated":                # the order of equal ids is free
            for key in ("pos", "vel", "rho"):
                assert np.array_equal(got[key], st[key][sel]), key
        import torch
        m = sel.size
        dev = [torch.zeros((m, 3), dtype=torch.float64, device="cuda"),
               torch.zeros((m, 3), dtype=torch.float32, device="cuda"),
               torch.zeros(m, dtype=torch.float32, device="cuda"),
               torch.zeros(m, dtype=torch.int32, device="cuda")]
        torch.cuda.synchronize()
        S.sph_subdomain_select(sim.ctx, mode, float(xlo), float(xhi), m, *dev)
        assert np.array_equal(dev[3].cpu().numpy().view(np.uint32), got["ids"])
        if ids != "repeated":
            for t, key in zip(dev, ("pos", "vel", "rho")):
                assert np.array_equal(t.cpu().numpy(), got[key]), key
    sim.check()
    sim.close()

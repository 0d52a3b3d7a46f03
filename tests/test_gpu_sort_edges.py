"""The radix sort around 128 tiles of 4,096 pairs (from where the tile counts are
scanned by a launch of their own) and around the 16 tiles whose counts a block
adds up at a time, on random, equal and few-valued keys, against numpy's stable
sort; every sort clears the scratch's error word."""
import numpy as np
import pytest

import __graft_entry__
from paper_1210_1017_gb300 import sph as S

pytestmark = pytest.mark.gpu
TILE = 4096


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    yield


@pytest.mark.parametrize("n", [5, TILE + 3, 15 * TILE + 1, 16 * TILE, 16 * TILE + 1, 127 * TILE + 9,
                               128 * TILE, 128 * TILE + 1, 131 * TILE - 1])
def test_sizes_around_the_dispatch(n):
    import torch
    rng = np.random.default_rng(n)
    vals = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    v = torch.from_numpy(vals.view(np.int32)).cuda()
    ko, vo = torch.empty_like(v), torch.empty_like(v)
    nb = int(S.lib().sph_radix_sort_scratch_bytes(n))
    scratch = torch.randint(0, 255, (nb,), dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    for bits, keys in ((32, rng.integers(0, 1 << 32, n, dtype=np.uint64)),
                       (24, np.full(n, 0x5a5a5a)), (16, rng.integers(0, 3, n) * 20000)):
        keys = keys.astype(np.uint32)
        k = torch.from_numpy(keys.view(np.int32)).cuda()
        order = np.argsort(keys, kind="stable")
        S.sph_radix_sort_selftest_timeout(scratch, nb, n, 4, st)
        with pytest.raises(S.SphError, match="SPH_ERR_TIMEOUT"):
            S.sph_radix_sort_status(scratch, nb, n, st)
        S.sph_radix_sort_pairs(k, v, ko, vo, n, bits, scratch, nb, st)
        S.sph_radix_sort_status(scratch, nb, n, st)
        assert np.array_equal(ko.cpu().numpy().view(np.uint32), keys[order])
        assert np.array_equal(vo.cpu().numpy().view(np.uint32), vals[order])

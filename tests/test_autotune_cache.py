"""The cached choice of the interaction shape is reused for a simulation of the
same size and density only: shapes differ by how many candidates they stage, so
another h/dp is tuned anew."""
import numpy as np

from paper_1210_1017_gb300 import cases
from paper_1210_1017_gb300 import sph as S


class _Sim:
    """A stand-in for Simulation: what autotune_cached looks at."""

    class torch:
        class cuda:
            @staticmethod
            def get_device_name(device):
                return "device"

    device, n_inst, ctx = 0, 1, None

    def __init__(self, h_over_dp, n=4000):
        case = cases.random_block(n, seed=1, h_over_dp=h_over_dp)
        self.n, self.P, self.taken = case.n, S.make_params(case.params(), 0.0), []

    def set_variant(self, v):
        self.taken.append(v)


def test_another_density_is_tuned_anew(monkeypatch, tmp_path):
    monkeypatch.setenv("XDG_CACHE_HOME", str(tmp_path))
    tuned = []

    def tune(ctx, reps):
        tuned.append(len(tuned))
        return tuned[-1], np.arange(16, dtype=np.float32)

    monkeypatch.setattr(S, "sph_autotune", tune)
    assert S.autotune_cached(_Sim(1.3))[0] == 0
    assert S.autotune_cached(_Sim(2.1))[0] == 1         # not the choice for 1.3
    again = _Sim(1.3)
    assert S.autotune_cached(again)[0] == 0 and again.taken == [0]
    again = _Sim(2.1)
    assert S.autotune_cached(again)[0] == 1 and again.taken == [1]
    assert S.autotune_cached(_Sim(1.3, 40000))[0] == 2  # another size, as before
    assert tuned == [0, 1, 2]

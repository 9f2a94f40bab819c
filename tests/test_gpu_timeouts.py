"""Every entry point of a context whose tensor-core products gave up reports DQMC_ETIMEOUT, not a singular matrix: the
fresh and the working G, G(tau), a sweep (whose stabilisation meets void matrices after the skipped products) and the
time-displaced measurement.  The waits end by their limit; another context then works on the same device."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_wrap", [4, 5])
def test_calls_after_a_wait_gave_up(n_wrap):
    from paper_1704_00131_gb300 import dqmc

    class Kept(dqmc.Ensemble):
        def close(self):
            pass

    m = W.ModelSpec(W.square_lattice(6, 6), U=4.0, dtau=0.1, L=20, n_wrap=n_wrap)
    ens = Kept.__new__(Kept)
    calls = {"init": lambda: ens.__init__([m], [0], precision="mixed_tc", seed=3, spin_limit=20000, tc_min_sites=1,
                                          test_stall=1),
             "greens": lambda: ens.greens(0, 0), "working": lambda: ens.greens(0, 1, fresh=False),
             "tau": lambda: ens.greens_tau(0, 0, 3), "sweep": lambda: ens.sweep(1),
             "greens after": lambda: ens.greens(0, 0), "measure_tau": lambda: ens.measure_tau(2)}
    for name, call in calls.items():
        with pytest.raises(dqmc.DqmcError) as e:
            call()
        assert e.value.status == dqmc.DQMC_ETIMEOUT, name
        assert "gave up" in str(e.value), name
    dqmc.Ensemble.close(ens)
    ok = dqmc.Ensemble([m], [0], precision="mixed_tc", seed=3, tc_min_sites=1)
    st = ok.sweep(1)
    assert 0 < st["accepted"] < st["proposals"] and np.isfinite(ok.greens(0, 0)[0]).all()
    ok.close()

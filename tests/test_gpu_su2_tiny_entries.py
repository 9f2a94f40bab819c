"""Reflectors whose leading entry is so small that its square is subnormal or zero (a site joined to the others by a
hopping of 1e-150 to 1e-170): G(0) and log|det| against the oracle, to the 1e-10 of the complex FP64 path."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [1e-150, 1e-158, 1e-160, 3e-161, 1e-170])
def test_leading_entry_with_a_subnormal_square(orc, h):
    from paper_1704_00131_gb300 import dqmc
    K = np.zeros((5, 5))
    K[:4, :4] = W.chain_lattice(4, mu=0.1)
    K[4, 4] = -3.0
    K[0, 4] = K[4, 0] = h
    dtau, U, L, nw = 0.1, 3.0, 6, 2
    f = W.random_fields(2, L, 5, seed=11)
    ens = dqmc.Su2Ensemble([dqmc.Su2Model(K, U=U, dtau=dtau, L=L, n_wrap=nw)], [0], fields=[f], seed=5)
    Go, lo, _ = orc.su2_green_udv(K, dtau, U, nw, f, 0)
    G, la, _, _ = ens.greens(0, fresh=False)
    assert np.abs(G - Go).max() < 1e-10
    assert la == pytest.approx(lo, rel=1e-10, abs=1e-10)
    ens.close()

"""The SU(2) kernels at the edges of their products' tiles (16 and 32) and below a warp: G(0), log|det| and the
trajectory of one sweep against the oracle, to the 1e-10 of the complex FP64 path."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [1, 2, 3, 15, 16, 17, 32, 33])
def test_su2_at_tile_edges(orc, sites):
    from paper_1704_00131_gb300 import dqmc
    K = W.chain_lattice(sites, mu=0.1, periodic=True)
    dtau, U, L, nw = 0.1, 3.0, 8, 4
    f = W.random_fields(2, L, sites, seed=sites)
    ens = dqmc.Su2Ensemble([dqmc.Su2Model(K, U=U, dtau=dtau, L=L, n_wrap=nw)], [0], fields=[f], seed=5)
    for _ in range(2):
        f = ens.get_fields()[0][0]
        Go, lo, ao = orc.su2_green_udv(K, dtau, U, nw, f, 0)
        G, la, ar, P = ens.greens(0, fresh=False)
        assert np.abs(G - Go).max() < 1e-10
        assert la == pytest.approx(lo, rel=1e-10, abs=1e-10)
        assert abs((ar - ao + np.pi) % (2 * np.pi) - np.pi) < 1e-10
        ens.sweep(1)
    ens.close()

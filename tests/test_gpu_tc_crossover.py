"""Around the site count from which DQMC_PREC_MIXED_TC chains take the tensor cores by default: the working
G(0) after a sweep against the FP64 oracle's on the swept fields, to the 1e-6 of the float-pair modes."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [71, 72, 73, 95])
def test_green_after_sweep(orc, sites):
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(W.chain_lattice(sites, mu=0.1, periodic=True), U=3.0, dtau=0.1, L=8, n_wrap=4)
    ens = dqmc.Ensemble([m], [0], precision="mixed_tc", seed=sites)
    ens.sweep(1)
    f, _ = ens.get_fields()
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    for s in (0, 1):
        Go, ldo, sgo = orc.green_udv(om, f[0], s, 0)
        G, ld, sg = ens.greens(0, s)
        assert np.abs(G - Go).max() < 1e-6 and sg == sgo
    ens.close()

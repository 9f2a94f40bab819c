"""The panelled pivoted QR, the LU and the solves at the edges of their panels (4 columns for the QR, 16 and
fewer for the LU) and at the smallest lattices: G(0) of freshly set fields against the FP64 oracle's, to the
1e-10 of the FP64 path and the 1e-6 of the float-pair one."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sites", [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 20, 21, 100, 160])
def test_green_at_panel_edges(orc, precision, sites):
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(W.chain_lattice(sites, mu=0.15, periodic=True), U=4.0, dtau=0.1, L=12, n_wrap=4)
    f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=100 + sites)
    ens = dqmc.Ensemble([m], [0], fields=[f], precision=precision)
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    for s in (0, 1):
        Go, ldo, sgo = orc.green_udv(om, f, s, 0)
        G, ld, sg = ens.greens(0, s)
        tol = 1e-10 if precision == "fp64" else 1e-6
        assert np.abs(G - Go).max() < tol
        assert ld == pytest.approx(ldo, rel=tol, abs=tol) and sg == sgo
    ens.close()


def test_uncoupled_sites_and_equal_columns(orc):
    """No hopping (every matrix diagonal, all column norms tied in pairs) and U = 0 (all norms tied)."""
    from paper_1704_00131_gb300 import dqmc
    for K, U in ((np.zeros((9, 9)), 4.0), (W.chain_lattice(9, periodic=True), 0.0)):
        m = W.ModelSpec(K, U=U, dtau=0.1, L=8, n_wrap=4)
        f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=8)
        ens = dqmc.Ensemble([m], [0], fields=[f], precision="fp64")
        om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
        for s in (0, 1):
            assert np.abs(ens.greens(0, s)[0] - orc.green_udv(om, f, s, 0)[0]).max() < 1e-10
        ens.close()

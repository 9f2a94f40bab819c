"""The exact-split tensor-core products of the FP64 kernels at the edges of their tiles (rows per tile
rounded to 16, 128 rows, 32 columns, 16-deep chunks) and around the size from which they run: the stable
G(0) against the FP64 oracle's, to the 1e-10 of the FP64 path (the products themselves are closer to
64-bit sums than FP64 ones)."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [31, 32, 33, 48, 63, 65, 97, 127, 128, 129, 161])
def test_fresh_green_at_tile_edges(orc, sites):
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(W.chain_lattice(sites, mu=0.1, periodic=True), U=3.0, dtau=0.1, L=8, n_wrap=4)
    f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=sites)
    ens = dqmc.Ensemble([m], [0], fields=[f], precision="fp64")
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    for s in (0, 1):
        Go, ldo, sgo = orc.green_udv(om, f, s, 0)
        for fresh in (False, True):
            G, ld, sg = ens.greens(0, s, fresh=fresh)
            assert np.abs(G - Go).max() < 1e-10
            assert ld == pytest.approx(ldo, rel=1e-10, abs=1e-10) and sg == sgo
    ens.close()


def test_wide_range_of_row_and_column_scales(orc):
    """A strong staggered potential spreads the rows and columns of the propagators over many powers of two."""
    from paper_1704_00131_gb300 import dqmc
    K = W.chain_lattice(40, periodic=True)
    K[np.arange(40), np.arange(40)] += np.linspace(-6.0, 6.0, 40)
    m = W.ModelSpec(K, U=2.0, dtau=0.1, L=12, n_wrap=2)
    f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=3)
    ens = dqmc.Ensemble([m], [0], fields=[f], precision="fp64")
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    for s in (0, 1):
        assert np.abs(ens.greens(0, s)[0] - orc.green_udv(om, f, s, 0)[0]).max() < 1e-10
    ens.close()

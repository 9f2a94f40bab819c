"""The QR where a block's entries leave the range of FP32 squares: four-valued fields, uniform in space up to a few
sites and opposite from block to block, so that one block scales by e^{+-44} or e^{+-66} while the whole product stays
of order one.  The columns' order (FP64) and the reflectors (float pairs) must not depend on that scale.

Tolerance: the FP64 G of these fields moves by at most 2e-12 when the blocks are shortened, hence the 1e-10 of the FP64
path; float pairs are asked for their 1e-6."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_tc"])
@pytest.mark.parametrize("sites,U,signs", [(20, 9.0, (1, -1, 1, -1)), (20, 20.0, (1, -1, 1, -1)),
                                           (20, 20.0, (1, -1, -1, 1)), (33, 20.0, (-1, 1, 1, -1))])
def test_green_of_blocks_of_opposite_scale(orc, precision, sites, U, signs):
    from paper_1704_00131_gb300 import dqmc
    nw, L = 20, 80
    big = np.random.default_rng(sites).random((L, sites)) >= 0.05
    f = (np.repeat(np.array(signs), nw)[:, None] * np.where(big, 2, 1)).astype(np.int8)
    m = W.ModelSpec(W.chain_lattice(sites, mu=0.1, periodic=True), U=U, dtau=0.1, L=L, n_wrap=nw, field_type=2)
    kw = {"tc_min_sites": 1} if precision == "mixed_tc" else {}
    ens = dqmc.Ensemble([m], [0], fields=[f], precision=precision, **kw)
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    tol = 1e-10 if precision == "fp64" else 1e-6
    for s in (0, 1):
        Go, ldo, sgo = orc.green_udv(om, f, s, 0)
        G, ld, sg = ens.greens(0, s, fresh=False)
        assert np.abs(G - Go).max() < tol
        assert ld == pytest.approx(ldo, rel=tol, abs=tol) and sg == sgo
    ens.close()

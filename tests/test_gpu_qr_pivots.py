"""Pivoting inside the panels of the QR where columns of a panel are nearly parallel: staggered fields at strong
coupling and long blocks, where the downdated norms of the float-pair panels cancel to rounding error of either sign.
G(0) of freshly set fields against the FP64 oracle's.

Tolerance: the FP64 G of these fields moves by at most 5e-14 when the blocks are shortened; the float-pair products
keep 42 bits, 2^11 times more, which gives 1e-10.  1e-9 is asked for, 1e-10 in FP64."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_tc"])
@pytest.mark.parametrize("lx,U,n_wrap,L,flips", [(2, 4.0, 20, 40, 0.05), (2, 4.0, 10, 40, 0.05), (6, 8.0, 10, 20, 0.0),
                                                 (6, 10.0, 10, 20, 0.0), (6, 12.0, 10, 20, 0.0),
                                                 (6, 12.0, 10, 20, 0.05)])
def test_green_of_staggered_fields(orc, precision, lx, U, n_wrap, L, flips):
    from paper_1704_00131_gb300 import dqmc
    N = lx * lx
    stag = np.array([1 if (x // lx + x % lx) % 2 else -1 for x in range(N)], dtype=np.int8)
    rng = np.random.default_rng(17)
    f = np.where(rng.random((L, N)) < flips, -stag, stag).astype(np.int8)
    m = W.ModelSpec(W.square_lattice(lx, lx), U=U, dtau=0.1, L=L, n_wrap=n_wrap)
    kw = {"tc_min_sites": 1} if precision == "mixed_tc" else {}
    ens = dqmc.Ensemble([m], [0], fields=[f], precision=precision, **kw)
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    tol = 1e-10 if precision == "fp64" else 1e-9
    for s in (0, 1):
        Go, ldo, sgo = orc.green_udv(om, f, s, 0)
        G, ld, sg = ens.greens(0, s, fresh=False)
        assert np.abs(G - Go).max() < tol
        assert ld == pytest.approx(ldo, rel=1e-9, abs=1e-9) and sg == sgo
    ens.close()

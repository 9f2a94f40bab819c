"""The windowed local updates at the edges of their windows (32 positions, 16 acceptances) and of the
delayed rank, against the oracle's sequential chain: fields and counts equal, G(0) within 1e-10 (FP64)
or 1e-6 (float pairs) of the oracle's."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_tc"])
@pytest.mark.parametrize("sites,vertices,delay,ft", [(31, 31, 16, 1), (32, 32, 15, 1), (33, 33, 17, 2), (65, 65, 64, 1),
                                                     (40, 33, 1, 2), (9, 1, 4, 1)])
def test_window_edges_match_the_sequential_chain(orc, precision, sites, vertices, delay, ft):
    from paper_1704_00131_gb300 import dqmc
    vs = np.random.default_rng(sites).permutation(sites)[:vertices].astype(np.int32)
    m = W.ModelSpec(W.chain_lattice(sites, mu=0.2, periodic=True), U=3.0, dtau=0.1, L=8, n_wrap=4, field_type=ft,
                    vertex_site=vs)
    ens = dqmc.Ensemble([m], [0, 0], precision=precision, delay_k=delay, seed=91)
    f0, _ = ens.get_fields()
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    chains = [orc.Chain(om, f0[c], seed=91, chain=c) for c in range(2)]
    sg = ens.sweep(2)
    so = [ch.sweep(2) for ch in chains]
    assert sg["accepted"] == sum(q.accepted for q in so) and sg["proposals"] == sum(q.proposals for q in so)
    fg, _ = ens.get_fields()
    for c, ch in enumerate(chains):
        assert np.array_equal(fg[c], ch.fields()[0])
        for s in (0, 1):
            assert np.abs(ens.greens(c, s)[0] - ch.green(s)).max() < (1e-10 if precision == "fp64" else 1e-6)
    ens.close()

"""Sweeps whose delayed vectors do not fit the shared memory (170 sites, rank 64: 2 x 64 x 172 entries of 8 bytes) and
lie in the chain's arena, where the float-pair flush stages them: against the oracle's sequential chain, fields and
counts equal, G(0) within 1e-10 (FP64) or 1e-6 (float pairs) of the oracle's, as for the windows."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dd_tile", [("fp64", 0), ("mixed", 0), ("mixed", 3), ("mixed", 4), ("mixed_tc", 0)])
def test_vectors_in_the_arena_match_the_sequential_chain(orc, precision, dd_tile):
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(W.chain_lattice(170, mu=0.2, periodic=True), U=3.0, dtau=0.1, L=4, n_wrap=2)
    ens = dqmc.Ensemble([m], [0], precision=precision, delay_k=64, seed=7, dd_tile=dd_tile)
    f0, _ = ens.get_fields()
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    ch = orc.Chain(om, f0[0], seed=7, chain=0)
    sg, so = ens.sweep(1), ch.sweep(1)
    assert sg["accepted"] == so.accepted and sg["proposals"] == so.proposals
    assert np.array_equal(ens.get_fields()[0][0], ch.fields()[0])
    for s in (0, 1):
        assert np.abs(ens.greens(0, s)[0] - ch.green(s)).max() < (1e-10 if precision == "fp64" else 1e-6)
    ens.close()

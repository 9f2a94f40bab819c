"""Sweeps of models with a single flavor (one CTA per chain, no peer to exchange blocks with) against the oracle's
sequential chain: fields and counts equal and G(0) within 1e-10 (FP64) or 1e-6 (float pairs) of the oracle's; in FP32,
whose rounding may change a decision, the wrapped G stays within 1e-3 of the fresh one."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed", "mixed_tc"])
@pytest.mark.parametrize("ft", [1, 2])
@pytest.mark.parametrize("sites,delay", [(7, 16), (33, 17), (65, 64)])
def test_one_flavor_matches_the_sequential_chain(orc, precision, ft, sites, delay):
    from paper_1704_00131_gb300 import dqmc
    K = W.chain_lattice(sites, mu=0.2, periodic=True)[None]
    m = W.ModelSpec(K, U=3.0, dtau=0.1, L=8, n_wrap=4, field_type=ft)
    kw = {"tc_min_sites": 1} if precision == "mixed_tc" else {}
    ens = dqmc.Ensemble([m], [0, 0], precision=precision, delay_k=delay, seed=19, **kw)
    f0, _ = ens.get_fields()
    sg = ens.sweep(2)
    fg, _ = ens.get_fields()
    if precision == "fp32":
        assert sg["prec_green_max"] < 1e-3
    else:
        om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
        chains = [orc.Chain(om, f0[c], seed=19, chain=c) for c in range(2)]
        so = [ch.sweep(2) for ch in chains]
        assert sg["accepted"] == sum(q.accepted for q in so) and sg["proposals"] == sum(q.proposals for q in so)
        for c, ch in enumerate(chains):
            assert np.array_equal(fg[c], ch.fields()[0])
            assert np.abs(ens.greens(c, 0)[0] - ch.green(0)).max() < (1e-10 if precision == "fp64" else 1e-6)
    ens.close()

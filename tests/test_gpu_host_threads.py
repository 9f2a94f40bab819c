"""Contexts of two host threads whose kernels want different shared memory (8 and 144 sites; SU(2) with 4 and 20): each
thread gets what a single thread gets, bit for bit."""
import threading

import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def results(sites, su2_sites, repeats):
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(W.chain_lattice(sites, mu=0.1, periodic=True), U=3.0, dtau=0.1, L=4, n_wrap=2)
    f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=sites)
    out = []
    for _ in range(repeats):
        ens = dqmc.Ensemble([m], [0], fields=[f], precision="fp64", seed=4)
        out += [ens.greens(0, 0, fresh=True)[0], ens.greens_tau(0, 1, 3), ens.measure_tau(2)[0]]
        out += list(ens.logdet_backward(0, f[None])) + list(ens.energy_backward(0, f[None]))
        ens.close()
        K = W.chain_lattice(su2_sites, mu=0.1, periodic=True)
        su = dqmc.Su2Ensemble([dqmc.Su2Model(K, U=3.0, dtau=0.1, L=4, n_wrap=2)], [0], seed=5)
        su.sweep(1)
        out += [su.get_fields()[0][0], su.greens(0, fresh=True)[0]]
        su.close()
    return [np.asarray(x).copy() for x in out]


def test_contexts_of_two_threads():
    sizes = ((8, 4), (144, 20))
    want = [results(a, b, 1) for a, b in sizes]
    got, failed = [None, None], []

    def work(i):
        try:
            got[i] = results(*sizes[i], 6)
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for i in range(2):
        assert len(got[i]) == 6 * len(want[i])
        for q, x in enumerate(got[i]):
            assert np.array_equal(x, want[i][q % len(want[i])])

"""Lattices at the limits of a CTA's shared memory (two and three stages of the split products, narrower QR panels, no
split products): G(0) of disconnected dimers against 2 x 2 products in numpy."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dimers(sites, mu=0.1):
    K = np.zeros((sites, sites))
    i = np.arange(0, sites - 1, 2)
    K[i, i + 1] = K[i + 1, i] = -1.0
    K[np.arange(sites), np.arange(sites)] = -mu
    return K


def dimer_green(m, f, s):
    """G(0) = (1 + B_L ... B_1)^-1 dimer by dimer."""
    N, lam = m.N, np.arccosh(np.exp(0.5 * m.dtau * m.U))
    G = np.zeros((N, N))
    for a in range(0, N, 2):
        idx = np.arange(a, min(a + 2, N))
        w, v = np.linalg.eigh(m.hopping[s][np.ix_(idx, idx)])
        E = (v * np.exp(-m.dtau * w)) @ v.T
        B = np.eye(len(idx))
        for t in range(m.L):
            B = E @ (np.exp(m.vertex_sign[s][idx] * lam * f[t][idx])[:, None] * B)
        G[np.ix_(idx, idx)] = np.linalg.inv(np.eye(len(idx)) + B)
    return G


@pytest.mark.parametrize("sites,precision", [(1105, "fp64"), (1105, "fp32"), (1104, "mixed"), (1296, "mixed_tc"),
                                             (1500, "mixed_tc"), (1561, "fp64"), (1735, "mixed")])
def test_green_of_large_lattices(sites, precision):
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(dimers(sites), U=4.0, dtau=0.2, L=2, n_wrap=1)
    f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=sites)
    ens = dqmc.Ensemble([m], [0], fields=[f], precision=precision)
    tol = {"fp64": 1e-10, "fp32": 1e-6}.get(precision, 1e-6)
    for s in (0, 1):
        G, _, _ = ens.greens(0, s, fresh=False)
        assert np.abs(G - dimer_green(m, f, s)).max() < tol
    ens.close()


def test_sweep_beyond_the_former_limit():
    from paper_1704_00131_gb300 import dqmc
    m = W.ModelSpec(dimers(1156), U=4.0, dtau=0.2, L=1, n_wrap=1)
    ens = dqmc.Ensemble([m], [0], precision="mixed", seed=3)
    st = ens.sweep(1)
    assert st["prec_green_max"] < 1e-6 and 0 < st["accepted"] < st["proposals"]
    f, _ = ens.get_fields()
    for s in (0, 1):
        assert np.abs(ens.greens(0, s, fresh=False)[0] - dimer_green(m, f[0], s)).max() < 1e-6
    ens.close()

"""The exact-split FP64 products on operands of wide range: site potentials that spread the rows of e^{-dtau K} over
2^20 (dtau W = 7) or those of a block of slices over 2^52 (n_wrap dtau W = 18), in rising, falling and mixed order of
the sites.  The split is fixed-point under the largest entry of a row of the left and a column of the right factor, so this
is where it could lose what FP64 sums keep.

Reference: G = (1 + B(beta, 0))^-1 in 70-digit decimals.  Tolerance: eight times the error of the FP64 oracle (plain
sums of FP64 products, unblocked QR) on the same fields, and 4 N 2^-52 where that error is a few units of 2^-52 itself.
In a CPU model of the chain the 63 bits of the split stay below it (1e-16 to 3e-15 beside 2e-15 to 8e-15 of the oracle
for sorted sites), and dropping what lies 2^40 below the largest entry exceeds it a hundredfold (3e-12 to 1e-10)."""
from decimal import Decimal, localcontext

import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _decimals(A):
    return np.array([[Decimal(float(x)) for x in row] for row in A], dtype=object)


def _exp(A, squarings=12, terms=16):
    A = A / Decimal(2 ** squarings)
    R = T = _decimals(np.eye(len(A)))
    for k in range(1, terms):
        T = T.dot(A) / Decimal(k)
        R = R + T
    for _ in range(squarings):
        R = R.dot(R)
    return R


def _inverse(A):
    n = len(A)
    M = np.concatenate([A, _decimals(np.eye(n))], axis=1)
    for k in range(n):
        p = max(range(k, n), key=lambda i: abs(M[i, k]))
        M[[k, p]] = M[[p, k]]
        M[k] = M[k] / M[k, k]
        for i in range(n):
            if i != k:
                M[i] = M[i] - M[k] * M[i, k]
    return M[:, n:]


def _exact_green(m, lam, fields, s):
    with localcontext() as ctx:
        ctx.prec = 70
        E = _exp(_decimals(m.hopping[s]) * Decimal(-m.dtau))
        B = _decimals(np.eye(m.N))
        for t in range(m.L):
            ev = [Decimal(0)] * m.N
            for k, i in enumerate(m.vertex_site):
                ev[i] += Decimal(float(m.vertex_sign[s][k] * lam * fields[t, k]))
            B = E.dot(np.array([x.exp() for x in ev], dtype=object)[:, None] * B)
        G = _inverse(_decimals(np.eye(m.N)) + B)
        return np.array([[float(x) for x in row] for row in G])


@pytest.mark.parametrize("sites,potential,L,n_wrap,order", [
    (33, 70.0, 4, 2, "rising"), (33, 70.0, 4, 2, "falling"), (33, 70.0, 4, 2, "mixed"),
    (33, 45.0, 8, 4, "rising"), (33, 45.0, 8, 4, "falling"), (65, 70.0, 4, 2, "rising"), (65, 70.0, 4, 2, "mixed")])
def test_green_of_wide_site_potentials(orc, sites, potential, L, n_wrap, order):
    from paper_1704_00131_gb300 import dqmc
    e = np.linspace(-potential, potential, sites)
    e = {"rising": e, "falling": e[::-1], "mixed": np.random.default_rng(5).permutation(e)}[order]
    K = W.chain_lattice(sites, periodic=True)
    K[np.arange(sites), np.arange(sites)] += e
    m = W.ModelSpec(K, U=3.0, dtau=0.1, L=L, n_wrap=n_wrap)
    f = W.random_fields(m.field_type, m.L, m.n_vertices, seed=3)
    ens = dqmc.Ensemble([m], [0], fields=[f], precision="fp64")
    om = orc.Model(m.hopping, m.vertex_site, m.vertex_sign, m.U, m.dtau, m.L, m.n_wrap, m.field_type)
    exact = [_exact_green(m, orc.ising_lambda(m.dtau, m.U), f, s) for s in (0, 1)]
    tol = 8 * max(np.abs(orc.green_udv(om, f, s, 0)[0] - exact[s]).max() for s in (0, 1)) + 4 * sites * 2.0 ** -52
    for s in (0, 1):
        for fresh in (False, True):
            assert np.abs(ens.greens(0, s, fresh=fresh)[0] - exact[s]).max() < tol
    ens.close()

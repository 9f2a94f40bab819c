"""The adjoints' workspace that a context keeps between calls: calls of growing and shrinking size and of
either kind leave nothing behind for the next one.  The kernels use no atomics, so that the same call of a
fresh context gives the same bits."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_kept_workspace_leaves_no_trace():
    from paper_1704_00131_gb300 import dqmc
    small = W.ModelSpec(W.square_lattice(3, 3, 1.0, 0.0, 0.1), U=3.0, dtau=0.1, L=8, n_wrap=4)
    large = W.ModelSpec(W.square_lattice(6, 6), U=4.0, dtau=0.1, L=12, n_wrap=4, field_type=2)
    kept = dqmc.Ensemble([small, large], [0, 1], precision="fp64")
    for index, n_cfg, kind in ((0, 1, "logdet"), (1, 3, "energy"), (0, 2, "energy"), (1, 1, "logdet"),
                               (1, 5, "logdet"), (0, 1, "logdet")):
        m = (small, large)[index]
        f = np.stack([W.random_fields(m.field_type, m.L, m.n_vertices, seed=7 + c) for c in range(n_cfg)])
        fresh = dqmc.Ensemble([small, large], [0, 1], precision="fp64")
        got = getattr(kept, f"{kind}_backward")(index, f)
        want = getattr(fresh, f"{kind}_backward")(index, f)
        fresh.close()
        for g, w in zip(got, want):
            assert np.array_equal(np.asarray(g), np.asarray(w))
    kept.close()

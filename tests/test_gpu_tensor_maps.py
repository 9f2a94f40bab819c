"""The adjoints write the tensor maps of each call over those of the last one, at the same addresses of the
workspace that the context keeps.  Models whose row tiles differ (36 sites: 48 rows; 100: 112; 130: two tiles of
80), alternated with equal numbers of configurations, give the bits that a fresh context gives."""
import numpy as np
import pytest

from paper_1704_00131_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_maps_of_alternating_models_at_one_address():
    from paper_1704_00131_gb300 import dqmc
    lat = (W.square_lattice(6, 6), W.square_lattice(10, 10), W.chain_lattice(130, mu=0.1, periodic=True))
    models = [W.ModelSpec(K, U=4.0, dtau=0.1, L=8, n_wrap=4) for K in lat]
    fields = [np.stack([W.random_fields(m.field_type, m.L, m.n_vertices, seed=31 + c) for c in range(2)])
              for m in models]
    want = {}
    for i in range(3):
        fresh = dqmc.Ensemble(models, [0, 1, 2], precision="fp64")
        for kind in ("logdet", "energy"):
            want[i, kind] = getattr(fresh, f"{kind}_backward")(i, fields[i])
        fresh.close()
    kept = dqmc.Ensemble(models, [0, 1, 2], precision="fp64")
    kept.energy_backward(2, fields[2])  # the largest: the block keeps its address from here on
    for i, kind in ((0, "logdet"), (1, "logdet"), (0, "energy"), (2, "logdet"), (1, "energy"), (0, "logdet"),
                    (1, "logdet"), (2, "energy")):
        got = getattr(kept, f"{kind}_backward")(i, fields[i])
        for g, w in zip(got, want[i, kind]):
            assert np.array_equal(np.asarray(g), np.asarray(w)), (i, kind)
    kept.close()

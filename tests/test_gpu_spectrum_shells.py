"""Shell binning of the spectrum at the edges of its rows: a row of n/2 + 1 modes is split over
warps of 32, so n = 61..66 has a row that ends just before, at and after a warp, and fewer bins
than shells drop the modes beyond. A field with energy in every mode, against the oracle.

Tolerances: FP64 sums and transforms, a few hundred roundings of 1.1e-16 per shell, and the
state's decoded velocity (1e-15 of 0.03): 1e-11 of a shell. FP32 velocities: 6e-8 each, 2e-5.
"""
import math

import numpy as np
import pytest

import oracle

from test_gpu_parity import lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,rel", [("f64", 1e-11), ("f32", 2e-5)])
@pytest.mark.parametrize("n,bins", [(4, 4), (5, 9), (61, 55), (62, 20), (63, 1), (64, 57),
                                    (65, 58), (66, 33)])
def test_shells_at_row_edges(kbc, storage, rel, n, bins):
    u = np.random.default_rng(n).uniform(-0.03, 0.03, (3, n, n, n))
    lat = lattice((n, n, n), nu=1e-3, storage=storage, scheme="pull")
    lat.init_field(None, u)
    E = lat.spectrum(bins)
    every = int(math.sqrt(3) * n / 2) + 2
    _, uu = oracle.macroscopic(lat.get_populations())
    ref = oracle.spectrum(uu, every)
    both = min(bins, every)
    assert E[0] == 0.0
    assert np.allclose(E[:both], ref[:both], rtol=rel, atol=rel * ref.max())
    assert not np.any(E[both:])

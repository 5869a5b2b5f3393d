"""Precision of recorded FP32 observables: at most 32 nodes are added up in
float, those of one or two rows of a tile; everything above is double."""
import numpy as np
import pytest

import oracle
import paper_1904_02471_gb300 as pkg

pytestmark = pytest.mark.gpu

VMAX4 = 2.33441421833897723932


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available()
    from paper_1904_02471_gb300 import build
    build.build()
    torch.cuda.init()


def test_rows_of_different_size_are_added_in_double():
    """Rows of density 1.5 and rows of 1 + 3 / 2^26, four by four: in float the
    sum of one node of each is off by 2^-26, in double by nothing. All of a
    node's deviation sits in one population, so that its density is exact."""
    nx, ny = 64, 64
    dr = np.where(np.arange(ny) // 4 % 2 == 0, 0.5, 3.0 * 2.0 ** -26)
    f = oracle.equilibrium(4, np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx)))
    f[5] += dr[:, None]
    dt = 0.1 / nx / VMAX4
    with pkg.Lattice("fd", 4, nx, ny, 2 * dt, dt=dt, precision="fp32") as L:
        L.config(2)
        L.set_populations(f)
        L.record(1, 4)
        L.step(1)
        first = L.series()[0]
    # the other populations' deviations are at most an ulp of their weights
    assert abs(first["mass"] - nx * (ny + dr.sum())) < nx * ny * (16 * 2.0 ** -55 + 2.0 ** -52)

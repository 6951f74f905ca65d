"""Jump-flood seeds against the oracle over grid sizes that take every column
length of the z-blocked pass, its read-ahead form, and its shortened candidate
sets (columns within a step of a side, whole lattices in a column), on dense,
sparse and single-triangle scenes."""
import numpy as np
import pytest

import oracle
from synth import scenes as S
from tests._util import seeds_to_linear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 8, 9, 12, 15, 17, 24, 31, 33, 47, 61, 64, 65, 75, 97, 130, 161, 200])
@pytest.mark.parametrize("tris", [1, 12, 3000])
def test_seeds_bit_exact(n, tris):
    from paper_2210_04449_gb300 import RTSDF
    m = S.random_soup(n, tris, size=0.02)
    rt = RTSDF(n)
    rt.set_tuning(jfa_tile=4)
    rt.upload_mesh(m.verts, m.tris)
    rt.voxelize()
    rt.jfa()
    rt.sync()
    occ = oracle.voxelize(m.verts, m.tris, np.zeros(3, np.float32), 1.0, n)
    want, _ = oracle.jfa(occ, n)
    assert np.array_equal(seeds_to_linear(rt.grids()["seeds"].cpu().numpy(), n), want)

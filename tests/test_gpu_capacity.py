"""Lists past what the int32 edge index holds, and images past what a packed edge holds."""
import numpy as np
import pytest

from gpu_util import assert_same_edges, lib_model
from oracle.neighbors import neighbor_list
from paper_2304_10061_gb300 import AllegroError
from synth import make_config, weights_to_blob

pytestmark = pytest.mark.gpu


# atoms in a cell of 0.62 Angstrom, every image of each within 4 Angstrom: about 2.5e9 edges (negative in
# int32), and about 4.5e9, which wrap to 2e8
@pytest.mark.parametrize("n", [1500, 2000])
def test_more_edges_than_the_index_holds(n):
    s, arch, w = make_config("c1")
    m = lib_model(weights_to_blob(arch, w))
    pos = np.random.default_rng(n).uniform(0.0, 0.62, (n, 3))
    with pytest.raises(AllegroError) as e:
        m.neighbors(pos, np.zeros(n, np.int32), np.eye(3) * 0.62)
    assert e.value.status == 4
    m.neighbors(s.pos, s.species, s.cell)
    assert_same_edges(m.get_neighbors(), neighbor_list(s.pos, s.cell, s.pbc, arch.r_c))
    m.close()


# images of a thin periodic axis: up to the 571st neighbour image along it, alone and across ordinary sizes
# of the other axes (a staged edge packs its image in 10 bits)
@pytest.mark.parametrize("n,width", [(1, 0.0085), (1, 0.0075), (2, 0.007), (7, 0.0071)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_thin_cells(axis, n, width):
    cell, pbc = np.eye(3) * 20.0, np.zeros(3, np.uint8)
    cell[axis, axis], pbc[axis] = width, 1
    rng = np.random.default_rng(n)
    pos = rng.uniform(0.0, 3.0, (n, 3))
    pos[:, axis] = rng.uniform(0.0, width, n)
    _, arch, w = make_config("c1")
    m = lib_model(weights_to_blob(arch, w))
    m.neighbors(pos, np.zeros(n, np.int32), cell, pbc)
    assert_same_edges(m.get_neighbors(), neighbor_list(pos, cell, pbc.astype(bool), arch.r_c))
    m.close()

"""Rows, columns and structures longer than the common ones: long cutoffs (a column holds 27 edges at 4
Angstrom, 90 at 6, 214 at 8, at the density of water) and batches of large structures.

Times are compared with those of other kernels, at margins of 1.5 or more on both sides, so they only
tell the forms apart."""
from dataclasses import replace

import numpy as np
import pytest

from gpu_util import assert_same_edges, lib_model
from oracle.neighbors import neighbor_list
from synth import ARCHS, lattice_box, make_weights, weights_to_blob

pytestmark = pytest.mark.gpu

C1 = ARCHS["c1"]


def _model(r_c=4.0):
    arch = replace(C1, r_c=r_c)
    return lib_model(weights_to_blob(arch, make_weights(arch, 0)))


def _kernel_us(m, call, name, passes=5):
    call()
    us = []
    for _ in range(passes):
        m.profile(True)
        call()
        us.append(m.profile_report()[0][name]["ms"] * 1e3)
        m.profile(False)
    return float(np.median(us))


# columns up to 4, 8 and more than 8 values per lane; cells likewise (the dense corner)
@pytest.mark.parametrize("r_c,n,dense", [(5.5, 700, 0), (6.0, 900, 0), (8.0, 1400, 0), (4.0, 600, 63), (4.0, 600, 64), (4.0, 600, 65),
                                         (4.0, 600, 129), (4.0, 600, 300)])
def test_long_columns(r_c, n, dense):
    """Lists, and the column sums that follow the column order: forces add up to zero and repeat bit for bit."""
    rng = np.random.default_rng(n + dense)
    s = lattice_box(n, max((n / 0.1) ** (1 / 3), 2.0 * r_c + 0.5), seed=n)
    pos = np.concatenate([s.pos, rng.uniform(0.1, 1.9, (dense, 3))]) if dense else s.pos
    types = (np.arange(len(pos)) % 2).astype(np.int32)
    m = _model(r_c)
    m.neighbors(pos, types, s.cell)
    assert_same_edges(m.get_neighbors(), neighbor_list(pos, s.cell, s.pbc, r_c))
    a = {k: v.cpu().numpy() for k, v in m.energy_forces().items()}
    m.neighbors(pos, types, s.cell)
    b = {k: v.cpu().numpy() for k, v in m.energy_forces().items()}
    m.close()
    for k in a:
        np.testing.assert_array_equal(a[k], b[k])
    # each edge's vector is added to one atom and taken from another: 1e-12 of the magnitudes, as elsewhere
    assert np.abs(a["F"].sum(0)).max() < 1e-12 * np.abs(a["F"]).sum()


@pytest.mark.parametrize("r_c", [6.0, 8.0])
def test_long_columns_are_not_sorted_by_one_lane(r_c):
    """262,144 atoms: the column passes take a fraction of the search's fill pass (1.7 and 4.2 times as
    long with a lane sorting a column, 0.33 and 0.52 with 16)."""
    s = lattice_box(262144, (262144 / 0.1) ** (1 / 3), seed=2)
    types = (s.species % 2).astype(np.int32)
    m = _model(r_c)
    call = lambda: m.neighbors(s.pos, types, s.cell)
    csc, fill = _kernel_us(m, call, "nb_csc"), _kernel_us(m, call, "nb_search_fill")
    m.close()
    print(f"r_c {r_c}: nb_csc {csc:.0f} us, nb_search_fill {fill:.0f} us")
    assert csc < 0.8 * fill, (csc, fill)

"""Rows, columns and structures longer than the common ones: long cutoffs (a column holds 27 edges at 4
Angstrom, 90 at 6, 214 at 8, at the density of water) and batches of large structures.

Times are compared with those of other kernels, at margins of 1.5 or more on both sides, so they only
tell the forms apart."""
from dataclasses import replace

import numpy as np
import pytest

from gpu_util import assert_same_edges, lib_model
from oracle.neighbors import neighbor_list
from paper_2304_10061_gb300 import AllegroError
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


# whole and part warps of a structure's atoms, one and many per lane
@pytest.mark.parametrize("sizes", [[255, 256, 257, 0, 1, 31, 33], [4001, 12, 2050]])
def test_batch_totals(sizes):
    """Totals of a batch are the sums of its atoms' energies; virials those of the structures by themselves."""
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    ss = [lattice_box(k, (k / 0.1) ** (1 / 3), seed=k) if k else None for k in sizes]
    pos = np.concatenate([s.pos for s in ss if s])
    types = np.concatenate([s.species % 2 for s in ss if s]).astype(np.int32)
    m = _model()
    m.neighbors_batched(offs, pos, types)
    out = {k: v.cpu().numpy() for k, v in m.energy_forces().items()}
    for b, s in enumerate(ss):
        Ea = out["E_atom"][offs[b]:offs[b + 1]]
        # the bound of the other sums here: 1e-12 of the magnitudes
        assert abs(out["E"][b] - Ea.sum()) <= 1e-12 * np.abs(Ea).sum()
        if s is None:
            assert out["E"][b] == 0 and not out["virial"][b].any()
            continue
        m.neighbors(s.pos, (s.species % 2).astype(np.int32))
        one = {k: v.cpu().numpy() for k, v in m.energy_forces().items()}
        # alone, a structure's rows come from the cell search: the order inside a row differs, so the
        # energies and forces agree to float32 rounding (2^-24 times about 10^2 terms)
        tol = 1e-5 * max(np.abs(one["virial"]).max(), 1e-30) + 1e-5 * np.abs(one["F"]).sum()
        assert np.abs(out["virial"][b] - one["virial"][0]).max() <= tol
    m.close()


def test_batch_of_large_structures():
    """Two structures of 60,000 atoms: a structure's sums are one block's, and testing each value on the
    float64 unit took them 626 us (a thread per atom and a tree, before, 306)."""
    n = 60000
    ss = [lattice_box(n, (n / 0.1) ** (1 / 3), seed=k) for k in (1, 2)]
    m = _model()
    m.neighbors_batched(np.array([0, n, 2 * n], np.int64), np.concatenate([s.pos for s in ss]),
                        np.concatenate([s.species % 2 for s in ss]).astype(np.int32))
    us = _kernel_us(m, m.energy_forces, "struct_reduce")
    m.close()
    print(f"struct_reduce {us:.0f} us")
    assert us < 400.0, us


def test_non_finite_energies_and_forces_are_reported():
    """Infinities and NaN are reported, the largest finite values are not."""
    def run(pos, sigma=None, mu=None, **kw):
        w = make_weights(C1, 0)
        for k, v in (("sigma", sigma), ("mu", mu)):
            if v is not None:
                w[k] = np.full_like(w[k], v)
        m = lib_model(weights_to_blob(C1, w))
        try:
            m.neighbors(np.asarray(pos, np.float64), np.zeros(len(pos), np.int32))
            m.energy_forces(**kw)
            return 0
        except AllegroError as e:
            return e.status
        finally:
            m.close()

    alone = [[0.0, 0.0, 0.0]]
    pair = [[0.0, 0.0, 0.0], [1.2, 0.0, 0.0]]
    assert run(pair) == 0
    assert run([[0.0, 0.0, 0.0], [0.0, 0.0, 0.0]]) == 6                     # NaN
    for big in (1.7e308, -1.7e308):   # the pair's model energy is -0.09 per atom: an infinity of either sign
        assert run(pair, sigma=-big, mu=1.05 * big, forces=False, virial=False) == 6
    for mu in (np.finfo(np.float64).max, -np.finfo(np.float64).max):
        assert run(alone, mu=mu) == 0
        assert run(alone, mu=mu, forces=False, virial=False) == 0

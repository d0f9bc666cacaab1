"""The forms a call can be dispatched to, at the sizes where one form ends and the next begins.

Neighbour lists are compared exactly with the oracle's rule, MLP widths with the oracle at the gates of
the precision, chunked and unchunked runs (which take different GEMM forms) bit for bit, and the
per-atom sums through two identities that hold to float64 rounding: the forces of a box add up to
zero (each edge's vector is added once and subtracted once), and the energies of an energy-only call
are those of a full call.  1e-12 of the sum of magnitudes is 10^4 times float64's rounding unit, above what
about 10^2 terms per atom accumulate.
"""
import ctypes

import numpy as np
import pytest
import torch

from gpu_util import BF16_F_RMS, FP32_E, FP32_F, FP32_W, assert_same_edges, errors, lib_model
from oracle.allegro import AllegroOracle
from oracle.neighbors import neighbor_list
from paper_2304_10061_gb300 import AllegroError
from synth import ARCHS, Arch, lattice_box, make_weights, weights_to_blob

pytestmark = pytest.mark.gpu

C1 = ARCHS["c1"]


def _box(n, seed=3):
    return lattice_box(n, max((n / 0.1) ** (1 / 3), 8.5), seed=seed)


@pytest.fixture(scope="module")
def model():
    m = lib_model(weights_to_blob(C1, make_weights(C1, 0)))
    yield m
    m.close()


def _check_rows(m, pos, cell, pbc, centers, types=None):
    """Sampled rows equal the oracle's; the whole list holds (j, i, -S) for every (i, j, S)."""
    types = np.zeros(len(pos), np.int32) if types is None else types
    m.neighbors(pos, types, cell, np.asarray(pbc, np.uint8))
    i, j, S = m.get_neighbors()
    assert_same_edges((i, j, S), (j, i, -np.asarray(S)))
    k = np.isin(i, centers)
    assert_same_edges((i[k], j[k], S[k]), neighbor_list(pos, cell, pbc, C1.r_c, centers=np.sort(centers)))


# a warp or a thread per centre, one scan launch or two, the cell and column tables of each
@pytest.mark.parametrize("pbc", [[1, 1, 1], [1, 0, 1]])
@pytest.mark.parametrize("n", [1, 31, 4095, 4097, 32767, 32769, 65536, 65537])
def test_neighbor_search_sizes(model, n, pbc):
    s = _box(n)
    c = np.random.default_rng(n).choice(n, min(n, 200), replace=False)
    _check_rows(model, s.pos, s.cell, pbc, c)


# cells and rows far beyond one warp's registers, alone and among many ordinary cells
@pytest.mark.parametrize("background", [0, 4000, 65600])
def test_neighbor_dense_cells(model, background):
    rng = np.random.default_rng(background)
    dense = rng.uniform(0.0, 8.0, (600, 3))
    pos, cell = dense, np.eye(3) * 40.0
    if background:
        s = _box(background)
        pos, cell = np.concatenate([s.pos, dense]), s.cell
    n = len(pos)
    c = np.concatenate([rng.choice(n, 64, replace=False), np.arange(n - 64, n)])
    _check_rows(model, pos, cell, [1, 1, 0], np.unique(c))


def test_list_outgrows_its_capacity():
    """Lists that overflow the room of the one before, and then shrink again, in one context."""
    m = lib_model(weights_to_blob(C1, make_weights(C1, 0)))
    for n, dens in ((64, 0.1), (300, 0.3), (2000, 0.1), (1500, 0.5), (5, 0.1), (6000, 0.1)):
        s = lattice_box(n, (n / dens) ** (1 / 3), seed=n)
        m.neighbors(s.pos, s.species % 2, s.cell)
        assert_same_edges(m.get_neighbors(), neighbor_list(s.pos, s.cell, s.pbc, C1.r_c))
        assert np.isfinite(m.energy_forces()["E"].item())
    m.close()


@pytest.mark.parametrize("shift", [4, 2])
def test_device_arrays_off_their_elements_alignment(model, shift):
    """Device arrays that start between two elements are copied, aligned ones are used in place: the same results."""
    s = _box(300)
    n, types = len(s.pos), (s.species % 2).astype(np.int32)
    L, ctx, st = model._L, model._ctx, lambda v: torch.tensor(np.frombuffer(v.tobytes(), np.uint8).copy(), device="cuda")
    want_edges = model.neighbors(torch.tensor(s.pos, device="cuda"), torch.tensor(types, device="cuda"), s.cell)
    want = {k: v.cpu().numpy() for k, v in model.energy_forces().items()}
    bufs = [torch.zeros(8 * k + 8, dtype=torch.uint8, device="cuda") for k in (3 * n, n, 1, n, 3 * n, 9)]
    bufs[0][shift:shift + 24 * n] = st(s.pos)
    bufs[1][shift:shift + 4 * n] = st(types)
    torch.cuda.synchronize()
    ptr = [b.data_ptr() + shift for b in bufs]
    cell, ne = np.ascontiguousarray(s.cell, np.float64), ctypes.c_int64(0)
    model._check(L.allegro_neighbors(ctx, n, ptr[0], ptr[1], cell.ctypes.data, None, ctypes.byref(ne)))
    assert ne.value == want_edges
    model._check(L.allegro_energy_forces(ctx, ptr[2], ptr[3], ptr[4], ptr[5]))
    for b, key in zip(bufs[2:], ("E", "E_atom", "F", "virial")):
        raw = b.cpu().numpy()[shift:shift + 8 * want[key].size].copy()
        np.testing.assert_array_equal(raw.view(np.float64), want[key].ravel())


@pytest.mark.parametrize("table", [None, [[4.0, 2.5], [3.0, 3.75]]])
def test_packed_molecules_without_cells(table):
    """Structures of 0 to 150 atoms, sizes around the lanes that share a centre."""
    sizes = [1, 0, 2, 15, 16, 17, 31, 32, 33, 0, 64, 65, 150, 3]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(4)
    pos = np.concatenate([rng.uniform(0, 2.0 + 1.5 * k ** (1 / 3), (k, 3)) for k in sizes])
    types = rng.integers(0, 2, offs[-1]).astype(np.int32)
    m = lib_model(weights_to_blob(C1, make_weights(C1, 0)))
    if table is not None:
        m.set_pair_cutoffs(np.array(table))
    m.neighbors_batched(offs, pos, types)
    want = []
    for b in range(len(sizes)):
        sl = slice(offs[b], offs[b + 1])
        if sizes[b] == 0:
            continue
        i, j, S = neighbor_list(pos[sl], None, [False] * 3, C1.r_c, species=types[sl], pair_rc=table)
        want.append((np.asarray(i) + offs[b], np.asarray(j) + offs[b], np.asarray(S).reshape(-1, 3)))
    assert_same_edges(m.get_neighbors(), tuple(np.concatenate(x) for x in zip(*want)))
    m.close()


# lanes per atom in the per-atom sums change at these sizes
@pytest.mark.parametrize("zbl", [False, True])
@pytest.mark.parametrize("n", [2999, 3001, 11999, 12001, 23999, 24001])
def test_atom_sums(model, n, zbl):
    s = _box(n, seed=n)
    model.set_zbl([1, 8] if zbl else None)
    model.neighbors(s.pos, s.species % 2, s.cell)
    full = {k: v.cpu().numpy() for k, v in model.energy_forces().items()}
    only = {k: v.cpu().numpy() for k, v in model.energy_forces(forces=False, virial=False).items()}
    model.set_zbl(None)
    assert np.abs(full["F"].sum(0)).max() < 1e-12 * np.abs(full["F"]).sum()
    np.testing.assert_allclose(only["E_atom"], full["E_atom"], rtol=0, atol=1e-12 * np.abs(full["E_atom"]).max())
    np.testing.assert_allclose(full["E"][0], full["E_atom"].sum(), rtol=0, atol=1e-12 * np.abs(full["E_atom"]).sum())


# widths: no multiple of four, eight or thirty-two; several column tiles, whole and ragged; the generic
# row path.  1500 atoms: enough tiles for CTA pairs, and row blocks in whole waves for the head epilogues of
# wide rows, the last block ragged; chunks of 2500 edges: too few for either
WIDTHS = {
    "odd": Arch(n_species=2, lmax=1, n_layers=2, channels=16, two_body=(18, 37), latent=(45, 33), edge=(7,)),
    "ragged_tiles": Arch(n_species=2, lmax=1, n_layers=2, channels=64, two_body=(60, 520), latent=(392, 328), edge=(12,)),
    "whole_tiles": Arch(n_species=2, lmax=1, n_layers=2, channels=64, two_body=(96, 512), latent=(768, 768), edge=()),
    "generic_whole_tiles": Arch(n_species=2, lmax=2, n_layers=3, channels=64, two_body=(64, 512), latent=(512,), edge=(16,)),
    "generic_128": Arch(n_species=2, lmax=2, n_layers=3, channels=32, two_body=(40, 128), latent=(128,), edge=()),
    "basis_12": Arch(n_species=2, lmax=2, n_layers=1, channels=8, two_body=(19, 32), latent=(32,), edge=(), n_bessel=12),
    "basis_1": Arch(n_species=2, lmax=2, n_layers=2, channels=8, two_body=(13,), latent=(30,), edge=(5,), n_bessel=1),
}
_REF = {}


def _reference(name):
    if name not in _REF:
        arch = WIDTHS[name]
        w = make_weights(arch, 21)
        s = _box(1500 if "tiles" in name else 330, seed=17)
        s.species = s.species % 2
        i, j, S = neighbor_list(s.pos, s.cell, s.pbc, arch.r_c)
        _REF[name] = (arch, w, s, AllegroOracle(arch, w).energy_forces(s.pos, s.species, s.cell, i, j, S))
    return _REF[name]


@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16", "fp8"])
@pytest.mark.parametrize("name", list(WIDTHS))
def test_mlp_widths(name, prec):
    arch, w, s, (E0, Ea0, F0, W0) = _reference(name)
    if (name, prec) == ("odd", "bf16"):
        # [x | s] with s at an odd column: no TMA box starts there, the call is refused
        m = lib_model(weights_to_blob(arch, w), precision=prec)
        m.neighbors(s.pos, s.species, s.cell)
        with pytest.raises(AllegroError):
            m.energy_forces()
        m.close()
        return
    runs = []
    for chunk in (0, 2500):
        m = lib_model(weights_to_blob(arch, w), precision=prec)
        if chunk:
            m.reserve(0, 0, 0, chunk)
        m.neighbors(s.pos, s.species, s.cell)
        runs.append({k: v.cpu().numpy() for k, v in m.energy_forces().items()})
        m.close()
    for r in runs:
        err = errors(r["E_atom"], r["F"], r["virial"][0], Ea0, F0, W0)
        if prec == "fp32":
            assert err["e_rel"] < FP32_E and err["f_max"] < FP32_F and err["w_rel"] < FP32_W, err
        else:
            # E4M3 products: 16 times the bfloat16 gates (three mantissa bits against seven)
            g = 16 if prec == "fp8" else 1
            assert err["f_rms"] < g * BF16_F_RMS and err["f_max"] < g * 10 * BF16_F_RMS, err
            assert err["e_rel"] < g * 1e-2 and err["w_rel"] < g * 5e-2, err
    if prec != "fp8":   # (FP8 scales each chunk's activations by themselves)
        for k in runs[0]:
            np.testing.assert_array_equal(runs[0][k], runs[1][k])

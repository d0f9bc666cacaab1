"""MLPs of one to five layers against the oracle, at the gates of the precision: the last layer's latent
MLP ends in an epilogue of its own on the BF16 path, and the layers before that pair are counted from it."""
import numpy as np
import pytest

from gpu_util import BF16_F_RMS, FP32_E, FP32_F, FP32_W, errors, lib_model
from oracle.allegro import AllegroOracle
from oracle.neighbors import neighbor_list
from synth import Arch, lattice_box, make_weights, weights_to_blob

pytestmark = pytest.mark.gpu


# channels x (l_max + 1) a multiple of 64 (K-concatenated heads) or not; layer pairs that fuse (widths of 64, 128
# and 256) and widths that run as single GEMMs
@pytest.mark.parametrize("layers,lmax,channels", [(1, 1, 32), (2, 2, 64), (2, 2, 32)])
@pytest.mark.parametrize("depth,widths", [(1, (64,)), (2, (256, 128)), (3, (256, 256, 256)), (3, (24, 72, 192)), (4, (256, 64, 256, 256)),
                                          (4, (40, 24, 192, 256)), (5, (64, 128, 256, 256, 256)), (5, (96, 16, 200, 32, 8))])
def test_depths(layers, lmax, channels, depth, widths):
    arch = Arch(n_species=2, lmax=lmax, n_layers=layers, channels=channels, two_body=widths, latent=widths, edge=(16,))
    w = make_weights(arch, 31 + depth)
    s = lattice_box(400, (400 / 0.1) ** (1 / 3), seed=depth)
    s.species = s.species % 2
    i, j, S = neighbor_list(s.pos, s.cell, s.pbc, arch.r_c)
    E0, Ea0, F0, W0 = AllegroOracle(arch, w).energy_forces(s.pos, s.species, s.cell, i, j, S)
    for prec in ("fp32", "tf32", "bf16"):
        m = lib_model(weights_to_blob(arch, w), precision=prec)
        m.neighbors(s.pos, s.species, s.cell)
        out = {k: v.cpu().numpy() for k, v in m.energy_forces().items()}
        only = m.energy_forces(forces=False, virial=False)["E_atom"].cpu().numpy()
        m.close()
        err = errors(out["E_atom"], out["F"], out["virial"][0], Ea0, F0, W0)
        if prec == "fp32":
            assert err["e_rel"] < FP32_E and err["f_max"] < FP32_F and err["w_rel"] < FP32_W, err
        else:
            # the gates hold for MLPs of two layers; roundings of more add up at most in proportion
            g = max(1.0, depth / 2)
            assert err["f_rms"] < g * BF16_F_RMS and err["f_max"] < g * 10 * BF16_F_RMS, (prec, err)
            assert err["e_rel"] < g * 1e-2 and err["w_rel"] < g * 5e-2, (prec, err)
        np.testing.assert_array_equal(only, out["E_atom"])
